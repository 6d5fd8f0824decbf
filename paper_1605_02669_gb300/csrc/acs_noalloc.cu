// acs_noalloc.cu -- acs_iterate_noalloc: one colony iteration on caller-owned
// device buffers that never allocates device memory.
//
// Some callers cannot call cudaMalloc: code that runs inside a memory pool
// or arena it does not own (an inference server that pre-reserves all device
// memory at start-up, a framework whose caching allocator must see every
// allocation), or code that must not allocate on its hot path. For them the
// per-iteration scratch of the construct kernel -- the visited bitmasks of
// all ants, the decay table P[k], the instance descriptor and the internal
// counters -- lives in one static device array of fixed size, kScratchBytes,
// that every GPU which loads this library keeps until the process exits.
#include <cuda_runtime.h>

#include <climits>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "acs.h"
#include "acs_device.cuh"
#include "acs_internal.cuh"

using namespace acs;

namespace {

constexpr size_t kScratchBytes = 4u << 20;   // 4 MiB per device
constexpr size_t kHeaderBytes = 256;         // descriptor, order, status, iteration, counters
constexpr size_t kTableBytes = 8192;         // decay table P[0..m], m <= 1024
constexpr size_t kVisOffset = kHeaderBytes + kTableBytes;
constexpr size_t kMaxVisWords = (kScratchBytes - kVisOffset) / 4;
constexpr int kMaxDevices = 64;

// The shared scratch. In host code this name is only a stand-in for the
// device array: its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

struct Header {
    InstDesc desc;
    int32_t order;
    int32_t status;
    int64_t iteration;
    unsigned long long stats[4];
};
static_assert(sizeof(Header) <= kHeaderBytes, "scratch header too large");

std::mutex g_mu;
unsigned char* g_addr[kMaxDevices] = {};

// Once per device, with that device current: look up the array's device address.
cudaError_t scratch_address(unsigned char** out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_scratch);
        if (e != cudaSuccess) return e;
        g_addr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_addr[dev];
    return cudaSuccess;
}

// One iteration of one instance by one CTA, eight lanes per ant, straight from
// the caller's rows and matrix: the construct kernel's packed rows, spatial
// order and lists of changed trails would not fit the fixed scratch (256 bytes
// per node and more). Per step: selections, the full scans of the ants whose
// candidates are used up (128-node items dealt to all warps), the folded local
// update. Same rules and bits as construct_kernel. The caller's coordinates are
// not limited to [0, 2^20), hence euc2d_wide().
constexpr int kLanes = 8;
constexpr int kPer = 32 / kLanes;

struct Shared {
    float* P;
    int *cur, *start, *nxt, *qant, *qc;
    long long* len;
    uint32_t* edge;              // (u << 16) | v
    unsigned long long* part;    // full-scan keys by queue entry
};

__host__ __device__ inline size_t shared_bytes(int m) { return 4u * ((size_t)m + 2) + 40u * (size_t)m + 64u; }

__device__ __forceinline__ bool seen(const uint32_t* vis, int j) { return (vis[j >> 5] >> (j & 31)) & 1u; }

__global__ void __launch_bounds__(1024, 1) iterate_kernel(const ConstructArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int qn, improved, bestant;
    __shared__ long long best_len;
    const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
    const int gl = lane & (kLanes - 1), gbase = lane & ~(kLanes - 1);
    const unsigned gmask = ((1u << kLanes) - 1u) << gbase;
    const int group = tid / kLanes, ngroups = nthr / kLanes, m = A.m;
    const InstDesc D = A.desc[0];
    const int n = D.n, cl = D.cl, W = D.W;
    const float tau0 = D.tau0;
    Shared S;
    {
        unsigned char* p = smem;
        S.len = (long long*)p; p += 8 * (size_t)m;
        S.part = (unsigned long long*)p; p += 8 * (size_t)m;
        S.cur = (int*)p; p += 4 * (size_t)m;
        S.start = (int*)p; p += 4 * (size_t)m;
        S.nxt = (int*)p; p += 4 * (size_t)m;
        S.qant = (int*)p; p += 4 * (size_t)m;
        S.qc = (int*)p; p += 4 * (size_t)m;
        S.edge = (uint32_t*)p; p += 4 * (size_t)m;
        S.P = (float*)p;
    }
    const int2* xy = reinterpret_cast<const int2*>(A.xy);
    uint32_t* vis_base = A.vis_global;
    float* tau = A.tau;
    int32_t *tours = A.tours, *best = A.best;
    const uint32_t it = (uint32_t)A.iteration[0];
    for (int i = tid; i <= m; i += nthr) S.P[i] = A.P[i];
    for (size_t i = tid; i < (size_t)m * W; i += nthr) vis_base[i] = 0u;
    if (tid == 0) best_len = __ldcg(A.best_len);
    __syncthreads();
    for (int a = tid; a < m; a += nthr) {   // step 0: first node (Alg. 1)
        const uint4 x = philox4x32_10(make_uint4(it, (uint32_t)a, 0u, 0u), A.key0, A.key1);
        const int start = (int)__umulhi(x.z, (uint32_t)n);
        S.cur[a] = S.start[a] = start;
        tours[(size_t)a * n] = start;
        vis_base[(size_t)a * W + (start >> 5)] |= 1u << (start & 31);
    }
    __syncthreads();
    int* const node[2] = {S.cur, S.nxt};   // node of ant a after step s: node[s & 1][a]
    for (int step = 1; step <= n; ++step) {
        if (tid == 0) qn = 0;
        __syncthreads();
        if (step < n) {
            for (int a = group; a < m; a += ngroups) {
                const int c = node[(step - 1) & 1][a];
                uint32_t* vis = vis_base + (size_t)a * W;
                int nv[kPer];
                float v[kPer];
                bool unv[kPer], any = false;
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    const int k = gl * kPer + i;
                    nv[i] = k < cl ? A.nn[(size_t)c * 32 + k] : 0;
                    unv[i] = k < cl && !seen(vis, nv[i]);
                    any |= unv[i];
                    v[i] = unv[i] ? __fmul_rn(__ldcg(tau + (size_t)c * n + nv[i]), A.w[(size_t)c * 32 + k]) : 0.0f;
                }
                if (!(__ballot_sync(gmask, any) & gmask)) {
                    if (gl == 0) {
                        const int q = atomicAdd(&qn, 1);
                        S.qant[q] = a;
                        S.qc[q] = c;
                        S.part[q] = 0ull;
                    }
                    continue;
                }
                const uint4 x = philox4x32_10(make_uint4(it, (uint32_t)a, (uint32_t)step, 0u), A.key0, A.key1);
                int first = -1, src;   // picked candidate of this lane, picked lane
                if (unit24(x.x) < A.q0) {
                    // Eq. 1: argmax, ties -> lowest rank
                    uint32_t mb = 0u;
#pragma unroll
                    for (int i = 0; i < kPer; ++i)
                        if (unv[i]) mb = max(mb, __float_as_uint(v[i]));
#pragma unroll
                    for (int off = kLanes / 2; off >= 1; off >>= 1)
                        mb = max(mb, __shfl_xor_sync(gmask, mb, off, kLanes));
#pragma unroll
                    for (int i = kPer - 1; i >= 0; --i)
                        if (unv[i] && __float_as_uint(v[i]) == mb) first = i;
                    src = __ffs(__ballot_sync(gmask, first >= 0) & gmask) - 1 - gbase;
                } else {
                    // Eq. 2: roulette over the inclusive scan of the 32 positions
                    float P[kPer];
#pragma unroll
                    for (int i = 0; i < kPer; ++i) P[i] = v[i];
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        float y[kPer];
#pragma unroll
                        for (int i = 0; i < kPer; ++i) {
                            const int dl = off >= kPer ? off / kPer : 1;
                            const float o = __shfl_up_sync(gmask, P[off >= kPer ? i : (i - off + kPer) % kPer], dl, kLanes);
                            if (off < kPer && i >= off) y[i] = __fadd_rn(P[i], P[i - off]);
                            else y[i] = gl >= dl ? __fadd_rn(P[i], o) : P[i];
                        }
#pragma unroll
                        for (int i = 0; i < kPer; ++i) P[i] = y[i];
                    }
                    const float t = __fmul_rn(unit24(x.y), __shfl_sync(gmask, P[kPer - 1], kLanes - 1, kLanes));
                    int last = -1, firstu = -1;
#pragma unroll
                    for (int i = 0; i < kPer; ++i) {
                        const bool pos = unv[i] && v[i] > 0.0f;
                        if (first < 0 && pos && P[i] > t) first = i;
                        if (pos) last = i;
                        if (firstu < 0 && unv[i]) firstu = i;
                    }
                    const unsigned bf = __ballot_sync(gmask, first >= 0) & gmask;
                    const unsigned bl = __ballot_sync(gmask, last >= 0) & gmask;
                    const unsigned bu = __ballot_sync(gmask, firstu >= 0) & gmask;
                    if (!bf) first = bl ? last : firstu;
                    src = bf ? __ffs(bf) - 1 - gbase : bl ? 31 - __clz(bl) - gbase : __ffs(bu) - 1 - gbase;
                }
                int mine = nv[0];
#pragma unroll
                for (int i = 1; i < kPer; ++i)
                    if (first == i) mine = nv[i];
                const int next = __shfl_sync(gmask, mine, src, kLanes);
                __syncwarp(gmask);
                if (gl == 0) {
                    node[step & 1][a] = next;
                    S.edge[a] = ((uint32_t)c << 16) | (uint32_t)next;
                    tours[(size_t)a * n + step] = next;
                    vis[next >> 5] |= 1u << (next & 31);
                }
            }
            __syncthreads();
            // Alg. 2's full scan of the queued ants
            const int E = qn, nch = (n + 127) >> 7;
            for (int item = tid >> 5; item < E * nch; item += nthr >> 5) {
                const int e = item / nch, ch = item - e * nch, c = S.qc[e];
                const uint32_t* vis = vis_base + (size_t)S.qant[e] * W;
                const int2 pc = xy[c];
                unsigned long long key = 0ull;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int j = (ch << 7) + i * 32 + lane;
                    if (j >= n || seen(vis, j)) continue;
                    const unsigned long long k2 =
                        pack_pj(__fmul_rn(__ldcg(tau + (size_t)c * n + j), heuristic(euc2d_wide(pc, xy[j]), A.beta)), j);
                    key = k2 > key ? k2 : key;
                }
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) {
                    const unsigned long long o = __shfl_xor_sync(0xffffffffu, key, off);
                    key = o > key ? o : key;
                }
                if (lane == 0 && key != 0ull) atomicMax(&S.part[e], key);
            }
            __syncthreads();
            for (int q = tid; q < E; q += nthr) {
                const int a = S.qant[q], c = S.qc[q];
                int next = (int)(0xffffffffu - (uint32_t)(S.part[q] & 0xffffffffull));
                if (S.part[q] == 0ull || next < 0 || next >= n) {
                    atomicExch(A.status, 4);   // no unvisited node: cannot happen before step n
                    next = c;
                }
                node[step & 1][a] = next;
                S.edge[a] = ((uint32_t)c << 16) | (uint32_t)next;
                tours[(size_t)a * n + step] = next;
                vis_base[(size_t)a * W + (next >> 5)] |= 1u << (next & 31);
            }
        } else {
            for (int a = tid; a < m; a += nthr)   // closing edges
                S.edge[a] = ((uint32_t)node[(step - 1) & 1][a] << 16) | (uint32_t)S.start[a];
        }
        __syncthreads();
        if (step % A.period) continue;
        // folded local update: the lowest ant on an edge stores both halves
        // from the trail every ant of the step chose on
        for (int a0 = 0; a0 < m; a0 += nthr) {
            const int a = a0 + tid;
            bool rep = a < m;
            int k = 0, u = 0, v = 0;
            float t = 0.0f;
            if (rep) {
                u = (int)(S.edge[a] >> 16);
                v = (int)(S.edge[a] & 0xffffu);
                const uint32_t fwd = S.edge[a], bwd = ((uint32_t)v << 16) | (uint32_t)u;
                for (int o = 0; o < m; ++o) {
                    const bool eq = S.edge[o] == fwd || S.edge[o] == bwd;
                    k += eq ? 1 : 0;
                    if (eq && o < a) rep = false;
                }
                if (rep) t = __ldcg(tau + (size_t)u * n + v);
            }
            if (rep) {
                const float t2 = local_rule(t, tau0, S.P[k]);
                tau[(size_t)u * n + v] = t2;
                tau[(size_t)v * n + u] = t2;
            }
        }
        __syncthreads();
    }
    // lengths, iteration best (ties -> lowest ant), best-so-far
    for (int a = group; a < m; a += ngroups) {
        const int32_t* t = tours + (size_t)a * n;
        long long sum = 0;
        for (int i = gl; i < n; i += kLanes) sum += euc2d_wide(xy[__ldcg(t + i)], xy[__ldcg(t + (i + 1 < n ? i + 1 : 0))]);
        __syncwarp(gmask);
#pragma unroll
        for (int off = kLanes / 2; off >= 1; off >>= 1) sum += __shfl_xor_sync(gmask, sum, off, kLanes);
        if (gl == 0) {
            S.len[a] = sum;
            A.lens[a] = sum;
        }
    }
    __syncthreads();
    if (tid < 32) {
        long long bl = 0x7fffffffffffffffll;
        int ba = 0x7fffffff;
        for (int a = tid; a < m; a += 32)
            if (S.len[a] < bl) { bl = S.len[a]; ba = a; }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) {
            const long long ol = __shfl_xor_sync(0xffffffffu, bl, off);
            const int oa = __shfl_xor_sync(0xffffffffu, ba, off);
            if (ol < bl || (ol == bl && oa < ba)) { bl = ol; ba = oa; }
        }
        if (tid == 0) {
            improved = bl < best_len;
            if (improved) best_len = bl;
            bestant = ba;
        }
    }
    __syncthreads();
    if (improved)
        for (int i = tid; i < n; i += nthr) best[i] = __ldcg(tours + (size_t)bestant * n + i);
    __syncthreads();
    const float delta = __double2float_rn(1.0 / (double)best_len);
    for (int i = tid; i < n; i += nthr) {
        const int u = __ldcg(best + i), v = __ldcg(best + (i + 1 < n ? i + 1 : 0));
        const float t2 = global_rule(__ldcg(tau + (size_t)u * n + v), delta, A.rho);
        tau[(size_t)u * n + v] = t2;
        tau[(size_t)v * n + u] = t2;
    }
    if (tid == 0) A.best_len[0] = best_len;
}

}  // namespace

extern "C" acs_status acs_iterate_noalloc(const int32_t* dev_coords, int32_t n,
                                          const int32_t* dev_nn32, const float* dev_w32,
                                          int32_t cl, float tau0, float* dev_tau,
                                          int32_t* dev_tours, int64_t* dev_lens,
                                          int32_t* dev_best, int64_t* dev_best_len,
                                          int64_t iteration, const acs_params* p, void* stream)
{
    if (!p || !dev_coords || !dev_nn32 || !dev_w32 || !dev_tau || !dev_tours || !dev_lens ||
        !dev_best || !dev_best_len)
        return ACS_EINVAL;
    if (n < 3 || n > kMaxN || cl < 1 || cl > kMaxCl || cl > n - 1 || iteration < 0)
        return ACS_EINVAL;
    if (p->m < 1 || p->m > kMaxM || p->beta < 0 || p->beta > 8) return ACS_EINVAL;
    if (!(p->q0 >= 0.0f && p->q0 <= 1.0f) || !(p->rho > 0.0f && p->rho < 1.0f) ||
        !(p->xi > 0.0f && p->xi < 1.0f))
        return ACS_EINVAL;
    if (p->memory != ACS_MEM_MATRIX || p->local_period < 1 || p->flags != 0) return ACS_EINVAL;
    if (!(tau0 > 0.0f)) return ACS_EINVAL;
    const int m = p->m;
    const int W = (n + 31) / 32;
    if ((size_t)m * (size_t)W > kMaxVisWords) return ACS_EINVAL;  // scratch too small
    if (4u * ((size_t)m + 1) > kTableBytes) return ACS_EINVAL;

    unsigned char* base = nullptr;
    cudaError_t e = scratch_address(&base);
    if (e != cudaSuccess) return ACS_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;

    Header h;
    std::memset(&h, 0, sizeof(h));
    h.desc.n = n;
    h.desc.cl = cl;
    h.desc.W = W;
    h.desc.instance = 0;
    h.desc.tau0 = tau0;
    h.order = 0;
    h.status = 0;
    h.iteration = iteration;
    std::vector<float> P(m + 1);
    const float f = 1.0f - p->xi;
    P[0] = 1.0f;
    for (int k = 1; k <= m; ++k) P[k] = P[k - 1] * f;

    // the kernel zeroes the visited words itself; the header (status and
    // counters included) and the table are rewritten on every call
    e = cudaMemcpyAsync(base, &h, sizeof(h), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(base + kHeaderBytes, P.data(), sizeof(float) * (m + 1),
                            cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return ACS_ECUDA;

    Header* dh = reinterpret_cast<Header*>(base);
    ConstructArgs A{};
    A.desc = &dh->desc;
    A.order = &dh->order;
    A.num_inst = 1;
    A.m = m;
    A.xy = dev_coords;
    A.nn = dev_nn32;
    A.w = dev_w32;
    A.tau = dev_tau;
    A.spm_idx = nullptr;
    A.spm_tail = nullptr;
    A.tours = dev_tours;
    A.lens = dev_lens;
    A.best = dev_best;
    A.best_len = dev_best_len;
    A.iteration = &dh->iteration;
    A.stats = dh->stats;
    A.vis_global = reinterpret_cast<uint32_t*>(base + kVisOffset);
    A.P = reinterpret_cast<const float*>(base + kHeaderBytes);
    A.status = &dh->status;
    A.q0 = p->q0;
    A.rho = p->rho;
    A.beta = p->beta;
    A.s = 0;
    A.period = p->local_period;
    A.skip_default = 0;
    A.key0 = (uint32_t)(p->seed & 0xffffffffull);
    A.key1 = (uint32_t)(p->seed >> 32);
    const size_t smem = shared_bytes(m);
    int block = m * kLanes < 64 ? 64 : (m * kLanes > 1024 ? 1024 : m * kLanes);
    block = (block + 31) / 32 * 32;
    e = cudaFuncSetAttribute(iterate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared_bytes(kMaxM));
    if (e != cudaSuccess) return ACS_ECUDA;
    iterate_kernel<<<1, block, smem, st>>>(A);
    if (cudaGetLastError() != cudaSuccess) return ACS_ECUDA;

    int32_t status = 0;
    e = cudaMemcpyAsync(&status, &dh->status, sizeof(status), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return ACS_ECUDA;
    return status == 0 ? ACS_OK : status == kWaitGaveUp ? ACS_ETIMEOUT : ACS_ECUDA;
}
