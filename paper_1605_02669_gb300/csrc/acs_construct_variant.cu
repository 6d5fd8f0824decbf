// acs_construct_variant.cu -- one variant of the construct kernel (all lane
// counts). Compiled once per variant, in parallel: ACS_MODE = 0 (matrix), 1
// (SPM, working copies in global memory), 2 (SPM, in shared memory); ACS_ALONE
// = 1 when every cluster is a single CTA; ACS_KIND = 0, 1, 2 for kShort, kLong and
// kTurns.
#include "acs_construct.cuh"

namespace acs {
template void* construct_variant<ACS_MODE, ACS_ALONE != 0, ACS_KIND>(int lanes);
}  // namespace acs
