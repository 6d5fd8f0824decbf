// acs_internal.cuh -- types shared by the host side and the kernels of libacs.
#pragma once
#include <cstdint>

namespace acs {

constexpr int kMaxCl = 32;          // candidate rows are padded to one warp
constexpr int kMaxN = 65536;        // nodes and positions in 16 bits each (edge keys, packed nodes)
constexpr int kMaxM = 1024;         // lists and the decay table in shared memory; 11-bit list entries (2 m)
constexpr int kCoordLimit = 1 << 20;

// Per-instance descriptor (device memory, read-only during a launch).
struct InstDesc {
    int32_t n;          // nodes
    int32_t cl;         // effective candidate width (<= 32, <= n-1)
    int32_t W;          // 32-bit visited words per ant = ceil(n/32)
    int32_t instance;   // Philox counter word 3
    int64_t xy_off;     // coords: xy[2*(xy_off + i) + {0,1}]
    int64_t row_off;    // candidate rows: nn/w[32*(row_off + c) + k]
    int64_t tau_off;    // matrix: tau[tau_off + c*n + j]; SPM: slot base spm_*[tau_off + c*s + i]
    int64_t node_off;   // per-node arrays (SPM tail, best tour): [node_off + c]
    int64_t tour_off;   // tours[tour_off + a*n + step]
    int64_t ant_off;    // lens[ant_off + a]
    int64_t vis_off;    // global visited words (when not in shared memory)
    int64_t hw_off;     // heuristic matrix hw[hw_off + c*n + j] (when present)
    float tau0;
    int32_t word_off;   // boxes of 32 spatially adjacent nodes: box[word_off + w], w < W
    int32_t dstrict;    // tau0 * eta^beta falls strictly with the distance from 1 to dstrict
    int32_t pad;
};

// Kernel arguments of the construct kernel (one iteration of Alg. 1 on every
// instance of a context).
struct ConstructArgs {
    const InstDesc* desc;
    const int32_t* order;     // instances in longest-first order
    int32_t num_inst;
    int32_t m;                // ants
    const int32_t* xy;
    const int32_t* nn;        // [rows][32], -1 padded
    const float* w;           // [rows][32], 0 padded
    const float* hw;          // heuristic matrix (relaxed mode only), or null
    // derived from the rows and the coordinates (read-only during a launch):
    // a packed node is (spatial position << 16) | index
    const uint2* rows;        // [rows][32] candidate rows: packed node, weight bits
    const uint32_t* spos;     // [rows] spatial position of each node
    const uint2* snode;       // [rows] by spatial position: x, y (20 bits each), index (16)
    const int4* box;          // per 32 positions: min x, min y, max x, max y
    float* tau;               // matrix entries, or SPM trail values
    int32_t* spm_idx;         // SPM neighbour per slot
    int32_t* spm_tail;        // SPM tail per node
    int32_t* tours;
    int64_t* lens;
    int32_t* best;            // best-so-far tours [sum n]
    int64_t* best_len;        // [B], INT64_MAX before the first iteration
    int64_t* iteration;       // [B]
    unsigned long long* stats;// [B][4]
    uint32_t* vis_global;     // visited words when they do not fit in smem
    const float* P;           // decay table P[0..m]
    int32_t* status;          // nonzero = an internal check failed
    float q0, rho;
    int32_t beta, s, period;
    uint32_t key0, key1;
    int32_t vis_in_smem, nodes_in_smem;
    int32_t max_n, max_w;     // largest instance: nodes, visited words (shared-memory layout)
    int32_t mc;               // ants per CTA of a cluster = ceil(m / cluster size)
    int32_t nrec;             // SPM records per CTA whose working copies are in shared memory
    int32_t skip_default;     // SPM: a local update of an absent edge inserts nothing
    const uint16_t* order_boxes; // [rows][kOrder] the boxes nearest to each node, by lower bound
                              // of the distance, 0xffff padded
    float* tauc;              // matrix: trails of the candidate rows [rows][32], kept equal to tau
    uint32_t* tl_node;        // matrix: per node the non-candidates whose trail is not tau0
    int32_t* tl_cnt;          // [rows][32] (packed), and how many; above kChanged: not listed
    const int32_t* asym;      // matrix, [B]: a restored matrix was not symmetric
    uint2* rec;               // SPM: the records' working copies (mode 1)
    unsigned long long wait_ns; // limit of one wait between the CTAs of a cluster
    int32_t hold;             // kHoldNone, or a test's barrier that never completes
    int32_t* sched;           // next-instance counter (zeroed before each launch) when the
                              // batch has more instances than resident clusters; null =
                              // cluster k takes instances k, k + clusters, ...
};

// Boxes listed per node for the search of the nearest unvisited node.
constexpr int kOrder = 32;
// Working copies of an SPM record on clusters of several CTAs.
constexpr int kCopies = 3;
// Threads of a CTA that shares an instance with others, without its publisher warp.
constexpr int kClusterAntThreads = 512;
// Device status of a wait that gave up (another CTA did not answer in kExchangeNs).
constexpr int kWaitGaveUp = 6;
constexpr unsigned long long kExchangeNs = 2000ull * 1000 * 1000;
// ConstructArgs::hold: the barrier of a ring that is made never to complete, by
// a test of the give-up.
constexpr int kHoldNone = 0, kHoldList = 1, kHoldStored = 2, kHoldPublished = 3;

// Time between two polls of a wait that counts towards its limit. A launch that
// does not run for a while (a shared GPU, a debugger) has one long poll; only
// time in which the wait was polled is held against the CTA waited for.
constexpr unsigned long long kPollNs = 10ull * 1000 * 1000;
__host__ __device__ inline unsigned long long counted_wait(unsigned long long last, unsigned long long now)
{
    const unsigned long long d = now > last ? now - last : 0ull;
    return d < kPollNs ? d : kPollNs;
}
// Changed non-candidate trails listed per node; a node with more (or with one
// below tau0, which only a restored state can hold) has its whole row read by
// the full scan.
constexpr int kChanged = 32;
constexpr int kReadAll = 1 << 20;

// Places of an edge list in shared memory: m rounded up to four per lane of a warp.
__host__ __device__ inline int list_places(int m) { return (m + 127) & ~127; }

// How the ants take their steps and look at a step's edge list: one ant per group
// that reads the list whole, four entries per lane at once (kShort) or in several
// goes (kLong); or in turns between barriers, with an index of the list (kTurns).
constexpr int kShort = 0, kLong = 1, kTurns = 2;
// A list's index (Colony): heads of chains by edge and by city, links.
__host__ __device__ inline int index_bits(int m)
{
    int b = 8;
    while ((1 << b) < 2 * m) ++b;
    return b;
}
__host__ __device__ inline uint32_t index_bytes(int m) { return (8u << index_bits(m)) + 14u * (uint32_t)list_places(m); }

// Shared-memory carve of the construct kernel; the same arithmetic runs on
// the host (to size the launch) and on the device (to place the arrays).
struct SmemLayout {
    uint32_t P, cur, start, len, edges, index, misc, box, rec, vis, nodes, total;
};

__host__ __device__ inline uint32_t align16(uint32_t x) { return (x + 15u) & ~15u; }

// mc = ants owned by one CTA of the cluster, m = ants of the instance, nrec =
// SPM records whose working copies (nc each) this CTA holds (0 = in global
// memory), s = SPM slots per record (0 for the matrix), indexed = with a list's
// index, nodes = nodes of the search's spatial order kept in shared memory (0 =
// read from global memory). Nothing before `box` depends on W.
__host__ __device__ inline SmemLayout smem_layout(int m, int mc, int nrec, int s, int W, int nc,
                                                  bool indexed, bool vis_in_smem, int nodes)
{
    SmemLayout L;
    uint32_t o = 0;
    L.P = o;     o = align16(o + 4u * (m + 1));
    L.cur = o;   o = align16(o + 4u * mc);
    L.start = o; o = align16(o + 4u * mc);
    L.len = o;   o = align16(o + 8u * mc);
    L.edges = o; o = align16(o + 4u * (s > 0 ? 4u : 8u) * (uint32_t)list_places(m));
    L.index = o; o = align16(o + (indexed ? index_bytes(m) : 0u));
    L.misc = o;  o = align16(o + 256u);
    L.box = o;   o = align16(o + 16u * (uint32_t)W);
    L.rec = o;   o = align16(o + 8u * (uint32_t)nc * (uint32_t)nrec * (uint32_t)(s + 1));
    L.vis = o;   if (vis_in_smem) o = align16(o + 4u * (uint32_t)mc * (((uint32_t)W + 3u) & ~3u));
    L.nodes = o; o = align16(o + 8u * (uint32_t)nodes);
    L.total = o;
    return L;
}

// What the learned-prior entry points need from a context (acs_api.cu).
struct CtxView {
    int n, cl;
    const int32_t* xy;   // coordinates of the instance [n][2]
    int32_t* nn;         // candidate rows [n][32]
    float* w;            // candidate weights [n][32]
    const int32_t* best; // best-so-far tour [n]
    void* stream;        // cudaStream_t of the context
    bool has_best;
};

}  // namespace acs
