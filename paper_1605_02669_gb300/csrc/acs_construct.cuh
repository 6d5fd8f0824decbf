// acs_construct.cuh -- the construct kernel: one full iteration of the Ant
// Colony System (Alg. 1) per instance, one thread-block cluster per instance.
//
// Mapping. The C CTAs of a cluster share one instance; CTA r owns ants
// r*mc .. r*mc+mc-1 (their visited bitmasks live in its shared memory). A
// group of L consecutive lanes builds one ant's tour; lane l of the group
// owns candidate ranks l*V .. l*V+V-1 (V = 32/L).
//
// What bounds it is the length of one step's dependent chain. A step is
//   select   Eq. 1 (argmax, q < q0) or Eq. 2 (Hillis-Steele roulette,
//            Sec. 3.1.1) over the unvisited candidates, whose trails are in
//            registers already;
//   push     the ant's edge (and, on the matrix, the trail it read) goes into
//            the step's edge list of every CTA of the cluster;
//   stage    the next city's candidate row, its visited bits and (matrix) its
//            trails are loaded while the lists travel. When every candidate is
//            visited the nearest unvisited node is looked for here (Alg. 2's
//            full scan, below);
//   fold     with the list complete, every group finds its own edge's
//            multiplicity k (an edge taken by k ants gets one folded local
//            update, Eq. 3 applied k times in closed form); the lowest ant on
//            an edge (matrix) or touching a record (SPM) stores the update.
//
// A list is looked over first (read_part(): four entries per lane, one vote);
// only when another ant's edge touches the ant's city are the entries taken one
// by one, in ant order. The code of a step is kept small: a lone warp's chain
// runs at about six cycles per instruction, and unrolled code of 170 KB at over
// ten.
//
// Clusters of several CTAs: the lists travel as asynchronous stores that
// complete a transaction count on the receiver's mbarrier (700-1260 cycles for
// 1 to 16 CTAs of 8 warps; a hardware cluster barrier with release and acquire
// takes 950-2000), and nothing else synchronises the ants. Updates are stored
// behind the next push and published behind the ants' backs: when all ants of
// a CTA have stored those of list k, its publisher warp tells every CTA, with
// release semantics. An ant stages its next city behind push k+1, when lists up
// to k are complete and updates up to k-1 are published, so it applies list k to
// what it reads there, and list k+1 when that is complete. (Two reads are outside
// this and wait for publication themselves: the whole-row read of a full scan and
// the closing edge's update.) Lists and mbarriers form a ring of four. An SPM
// record has three copies, each with the number of the update that wrote it;
// update k goes to the copy after the latest, so the copy published by k-1 stays
// whole while k and k+1 are being stored.
//
// One CTA per instance ("alone"): two CTA barriers a step, one after the push
// and one after the stores, about 100 cycles each; every read is then current
// and comes from L1 when it can.
//
// In turns (construct_turns_kernel): barriers on both sides of the updates, and
// groups of 8 or 16 lanes that take several ants when a CTA has more. The step's
// edges are looked up in hash chains, and a thread replays a record's events. It
// serves CTAs with more ants than groups, and colonies in which an ant meets so
// many others that reading lists costs more than the barriers (step_kind()).
//
// Measured (ms per iteration; before: a kernel with two cluster barriers a step
// and CTA-wide scans): n = 1002 and 2392, m = 128, matrix 13.1 to 5.2, SPM 18.4 to
// 6.7; eight of n = 10000 and eight of 20000, m = 256, matrix 348 to 99, SPM 252 to
// 159; 256 of n <= 2500, matrix and SPM, m = 64 21.2 to 10.4 and 26.2 to 13.4, m =
// 256 50 to 30 and 66 to 34.
//
// Alg. 2's full scan (the best of all unvisited nodes when the candidates are
// used up): every node that no best tour has used has trail tau0, so the scan
// is a search for the nearest unvisited node, plus the few nodes whose trail
// differs (matrix: the row's list of non-candidate nodes with a changed
// trail; SPM: the record). The search goes through bounding boxes of 32 nodes
// that follow each other on a Hilbert curve (bit i of visited word w is the
// i-th node of box w), in the order of the city's list of nearest boxes.
// Boxes and, when they fit, nodes are in shared memory.
//
// Mutable global state is written by one SM and read by others, so clusters
// read it with L2-coherent loads (ld.global.cg).
#pragma once
#include <climits>
#include <cstdint>
#include <type_traits>

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "acs_device.cuh"
#include "acs_internal.cuh"

namespace cg = cooperative_groups;

namespace acs {

namespace {

constexpr uint32_t kNoCity = 0xffffffffu;
constexpr uint32_t kNoEdge = 0u;   // the key of no edge (its ends would be the same city)
constexpr int kAloneThreads = 1024;
constexpr int kClusterThreads = kClusterAntThreads + 32;   // with the publisher warp
constexpr int kRing = 4;   // edge lists (and mbarriers) in flight, a power of two
struct Misc {
    int improved;
    int bestant;
    unsigned long long stat[3];   // fallback, spm hits, spm misses
    long long best_len;
    long long iteration;
    int next;                     // the cluster's next instance (drawn by rank 0)
    int next_local;               // this CTA's copy of rank 0's draw
    int stop;                     // a wait of this cluster gave up
    unsigned long long bar[kRing];   // completion of each list
    unsigned long long sdone[kRing]; // this CTA's updates of a list are stored
    unsigned long long pub[kRing];   // every CTA's updates of a list are published
};
static_assert(sizeof(Misc) <= 256, "misc block of the shared-memory layout");

__device__ __forceinline__ uint32_t node_id(uint32_t p) { return p & 0xffffu; }
__device__ __forceinline__ uint32_t edge_key(uint32_t u, uint32_t v)
{
    return (min(u, v) << 16) | max(u, v);
}
__device__ __forceinline__ bool touches(uint32_t key, uint32_t c)
{
    return ((key >> 16) == c || (key & 0xffffu) == c) && key != kNoEdge;
}
// the end of edge `key` that is not c
__device__ __forceinline__ uint32_t other_end(uint32_t key, uint32_t c)
{
    return (key >> 16) == c ? (key & 0xffffu) : (key >> 16);
}

__device__ __forceinline__ bool visited(const uint32_t* vis, uint32_t pos)
{
    return (vis[pos >> 5] >> (pos & 31)) & 1u;
}

// ---- a group of L lanes
//
// Every collective is executed by the whole warp (full mask), groups without
// work going along under a predicate: a ballot with a mask of its own per
// group took 289 cycles, one over the warp takes 27 (shuffles 43 and 38).

__device__ __forceinline__ bool any_lane(bool p) { return __any_sync(0xffffffffu, p); }
template <int L>
struct Group {
    int gl;          // lane within the group
    int gbase;       // the group's first lane

    __device__ __forceinline__ explicit Group(int lane) : gl(lane & (L - 1)), gbase(lane & ~(L - 1)) {}
    // p, the same on all lanes of a group, for any group of the warp
    __device__ __forceinline__ bool any_group(bool p) const
    {
        if constexpr (L == 32) return p;
        else return any_lane(p);
    }
    // lanes with p, bit i = lane i of the group
    __device__ __forceinline__ unsigned ballot(bool p) const
    {
        const unsigned b = __ballot_sync(0xffffffffu, p);
        if constexpr (L == 32) return b;
        else return (b >> gbase) & ((1u << (L & 31)) - 1u);
    }
    template <typename T>
    __device__ __forceinline__ T shfl(T v, int src) const
    {
        return __shfl_sync(0xffffffffu, v, src, L);
    }
    template <typename T>
    __device__ __forceinline__ T shfl_up(T v, int d) const
    {
        return __shfl_up_sync(0xffffffffu, v, d, L);
    }
    __device__ __forceinline__ uint32_t max_u32(uint32_t v) const
    {
        if constexpr (L == 32) {
            v = __reduce_max_sync(0xffffffffu, v);
        } else if constexpr (L >= 8) {
            // a whole-warp reduction per group: 22 cycles each, pipelined,
            // where a shuffle and a maximum take 42, four or three times over
            uint32_t r = 0u;
#pragma unroll
            for (int g = 0; g < 32; g += L) {
                const uint32_t x = __reduce_max_sync(0xffffffffu, gbase == g ? v : 0u);
                r = gbase == g ? x : r;
            }
            v = r;
        } else {
#pragma unroll
            for (int off = L / 2; off >= 1; off >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, off, L));
        }
        return v;
    }
    __device__ __forceinline__ uint32_t min_u32(uint32_t v) const { return ~max_u32(~v); }
    __device__ __forceinline__ uint32_t add_u32(uint32_t v) const
    {
        if constexpr (L == 32) {
            v = __reduce_add_sync(0xffffffffu, v);
        } else if constexpr (L >= 8) {
            uint32_t r = 0u;
#pragma unroll
            for (int g = 0; g < 32; g += L) {
                const uint32_t x = __reduce_add_sync(0xffffffffu, gbase == g ? v : 0u);
                r = gbase == g ? x : r;
            }
            v = r;
        } else {
#pragma unroll
            for (int off = L / 2; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off, L);
        }
        return v;
    }
    // maximum of the packed full-scan keys: the largest product bits, then the
    // largest low word among the lanes that hold them
    __device__ __forceinline__ unsigned long long max_key(unsigned long long k) const
    {
        const uint32_t hi = (uint32_t)(k >> 32);
        const uint32_t mh = max_u32(hi);
        const uint32_t ml = max_u32(hi == mh ? (uint32_t)k : 0u);
        return ((unsigned long long)mh << 32) | ml;
    }
};

// V consecutive candidates of a row: packed nodes and weights
template <int V>
__device__ __forceinline__ void load_row(const uint2* row, uint32_t (&nv)[V], float (&wv)[V])
{
    if constexpr (V == 1) {
        const uint2 a = __ldg(row);
        nv[0] = a.x;
        wv[0] = __uint_as_float(a.y);
    } else {
#pragma unroll
        for (int i = 0; i < V; i += 2) {
            const uint4 a = __ldg(reinterpret_cast<const uint4*>(row + i));
            nv[i] = a.x;
            wv[i] = __uint_as_float(a.y);
            nv[i + 1] = a.z;
            wv[i + 1] = __uint_as_float(a.w);
        }
    }
}

// V consecutive trails of a row
template <int V>
__device__ __forceinline__ void load_trails(const float* row, bool alone, float (&tv)[V])
{
    if constexpr (V == 1) {
        tv[0] = alone ? *row : __ldcg(row);
    } else if constexpr (V == 2) {
        const float2* p = reinterpret_cast<const float2*>(row);
        const float2 a = alone ? *p : __ldcg(p);
        tv[0] = a.x;
        tv[1] = a.y;
    } else {
#pragma unroll
        for (int i = 0; i < V; i += 4) {
            const float4* p = reinterpret_cast<const float4*>(row + i);
            const float4 a = alone ? *p : __ldcg(p);
            tv[i] = a.x;
            tv[i + 1] = a.y;
            tv[i + 2] = a.z;
            tv[i + 3] = a.w;
        }
    }
}

// ---- Alg. 2's full scan as a search over boxes of 32 nodes

// Squared distance from p to box b, in FP32: at most 2^-22 above the exact
// value (the differences are below 2^20 and exact; two products and a sum).
__device__ __forceinline__ float box_bound(int4 b, int2 p)
{
    const float dx = (float)max(max(b.x - p.x, p.x - b.z), 0);
    const float dy = (float)max(max(b.y - p.y, p.y - b.w), 0);
    return __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
}

// Node of the spatial order in eight bytes: x and y (20 bits each), index.
__device__ __forceinline__ int2 node_point(uint2 q)
{
    return make_int2((int)(q.x & 0xfffffu), (int)((q.x >> 20) | ((q.y & 0xffu) << 12)));
}

// The search by full-scan keys for the groups with `on`: every unvisited node
// (of the boxes closer than three units when `close`: distances 0 and 1 have
// one weight).
template <int L>
__device__ __noinline__ uint32_t nearest_by_key(int lane, int2 pc, int W, const uint32_t* vis, const uint2* nodes,
                                                const int4* box, float tau0, int beta, bool close, bool on)
{
    const Group<L> G(lane);
    unsigned long long key = 0ull;
#pragma unroll 1
    for (int w = G.gl; on && w < W; w += L) {
        uint32_t free = ~vis[w];
        if (free && close && box_bound(box[w], pc) > 9.0f) free = 0u;
#pragma unroll 1
        while (free) {
            const uint2 q = nodes[w * 32 + __ffs(free) - 1];
            free &= free - 1u;
            const unsigned long long k2 =
                pack_pj(__fmul_rn(tau0, heuristic(euc2d(pc, node_point(q)), beta)), (int)(q.y >> 16));
            key = k2 > key ? k2 : key;
        }
    }
    __syncwarp();
    return 0xffffffffu - (uint32_t)G.max_key(key);
}

// The boxes of a city's list: lane l of a group holds entries l*N .. l*N+N-1.
template <int L>
struct Order {
    static constexpr int N = kOrder / L;
    static constexpr int Q = (N + 3) / 4;
    uint2 q[Q];
    __device__ __forceinline__ void load(const uint16_t* row, int gl)
    {
        if constexpr (N == 1) {
            q[0].x = __ldg(row + gl);
        } else if constexpr (N == 2) {
            q[0].x = __ldg(reinterpret_cast<const uint32_t*>(row) + gl);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) q[i] = __ldg(reinterpret_cast<const uint2*>(row) + gl * Q + i);
        }
    }
    __device__ __forceinline__ int entry(int i) const
    {
        if constexpr (N == 1) return (int)q[0].x;
        uint2 x = q[0];
#pragma unroll
        for (int j = 1; j < Q; ++j)
            if (i >> 2 == j) x = q[j];
        return (int)(((N > 2 && (i & 2) ? x.y : x.x) >> (16 * (i & 1))) & 0xffffu);
    }
};

// For the groups with `need`: the unvisited node with the largest full-scan
// key of trail tau0, i.e. the lowest node among those with the largest product
// tau0 * eta^beta. The city's kOrder nearest boxes come from its list; boxes
// with an unvisited node and a lower bound that the best distance does not
// exclude are evaluated by the whole group, a lane per node. When the list's
// last box is not excluded either, all boxes are gone through. Between 2 and
// dstrict the product falls strictly with the distance, so the nearest node,
// ties to the lowest index, is the one; elsewhere keys decide. Returned as
// (index << 16) | spatial position: nothing is looked up behind the search.
template <int L>
__device__ __forceinline__ uint32_t nearest_unvisited(const Group<L>& G, const Order<L>& order, int2 pc, int W,
                                                      const uint32_t* vis, const uint2* nodes, const int4* box,
                                                      const uint32_t* spos, float tau0, int beta, int dstrict,
                                                      bool need)
{
    const float inf = __int_as_float(0x7f800000);
    uint32_t d = 0xffffffffu, at = 0xffffffffu, md = 0xffffffffu;   // at: index and position
    float thr = inf;    // nodes of a box whose bound exceeds thr are farther than md + 1
    constexpr int N = Order<L>::N;
    bool live = need;
#pragma unroll 1
    for (int i = 0; G.any_group(live); ++i) {
        int w = i < N ? order.entry(i) : (i - N) * L + G.gl;
        const bool in = live && w < W;   // 0xffff pads the list of fewer boxes
        if (!in) w = 0;
        const uint32_t word = in ? vis[w] : 0xffffffffu;
        const float x = in ? box_bound(box[w], pc) : inf;
        unsigned q = G.ballot(word != 0xffffffffu && x <= thr);
        // several boxes at once: a search needs three or four, and a box alone
        // is a chain of 350 cycles
        constexpr int B = L >= 16 ? L / 8 : 1;
#pragma unroll 1
        while (G.any_group(q != 0u)) {
            uint2 nd[B][32 / L];
            uint32_t free[B], pos[B];
#pragma unroll
            for (int e = 0; e < B; ++e) {
                const int src = q ? __ffs(q) - 1 : 0;
                const uint32_t bits = ~G.shfl(word, src);
                const int we = G.shfl(w, src);
                free[e] = q ? bits : 0u;
                q &= q - 1u;
                pos[e] = (uint32_t)(we * 32 + G.gl);
#pragma unroll
                for (int j = 0; j < 32 / L; ++j)
                    if ((free[e] >> (j * L + G.gl)) & 1u) nd[e][j] = nodes[pos[e] + j * L];
            }
#pragma unroll
            for (int e = 0; e < B; ++e)
#pragma unroll
                for (int j = 0; j < 32 / L; ++j)
                    if ((free[e] >> (j * L + G.gl)) & 1u) {
                        const uint32_t dd = (uint32_t)euc2d(pc, node_point(nd[e][j]));
                        const uint32_t x = (nd[e][j].y & 0xffff0000u) | (pos[e] + j * L);
                        if (dd < d || (dd == d && x < at)) {
                            d = dd;
                            at = x;
                        }
                    }
            __syncwarp();
            md = G.min_u32(d);
            if (md != 0xffffffffu) {
                const float r = (float)(md + 2u);
                thr = r * r * 1.000001f;
            }
            q &= G.ballot(x <= thr);
        }
        const float last = G.shfl(x, L - 1);
        if (i == N - 1 && (W <= kOrder || last > thr)) live = false;   // so are the boxes that are not listed
        if (i >= N && (i - N + 1) * L >= W) live = false;
    }
    uint32_t best = G.min_u32(d == md ? at : 0xffffffffu);
    const bool keys = need && !(md >= 2u && (int)md < dstrict);
    if (G.any_group(keys)) {
        const uint32_t bk = nearest_by_key<L>(G.gbase + G.gl, pc, W, vis, nodes, box, tau0, beta,
                                              md < 2u && dstrict > 2, keys);
        if (keys) best = bk > 0xffffu ? 0u : (bk << 16) | __ldg(spos + bk);
    }
    return best;
}

// ---- SPM records: NC copies of s slots and the tail. rec[q*NC + i] =
// {node, trail bits} of slot q < s in copy i; rec[s*NC + i] = {tail, number of
// the update that wrote the copy}. NC = 3 on clusters, 1 in a CTA alone.

// A group's private copy of one record: lane l holds slots l, l + L, ...
template <int V>
struct Record {
    int32_t idx[V];
    float val[V];
    int tail;
    int buf;    // the copy that holds the latest state
};

// ---- exchange of edge lists between the CTAs of a cluster

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t remote_addr(uint32_t a, int rank)
{
    uint32_t o;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(rank));
    return o;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, int arrivals)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// stores that count towards the receiver's mbarrier when they land
__device__ __forceinline__ void st_async(uint32_t at, uint32_t bar, uint2 v)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(at),
                 "r"(v.x), "r"(v.y), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async(uint32_t at, uint32_t bar, uint32_t v)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(at), "r"(v),
                 "r"(bar)
                 : "memory");
}
// Whether phase `parity` has completed. Acquire at cluster scope: what the
// barriers order (lists in shared memory, trails and records) was written by
// other CTAs and released at that scope; the default would be the CTA's.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0u;
}
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Waits for phase `parity` of the barrier; false when it has not completed
// within `limit` ns of counted time, or another wait of the cluster gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, unsigned long long limit,
                                          const volatile int* stop)
{
    unsigned long long last = global_ns(), spent = 0ull;
    while (!mbar_test(bar, parity)) {
        const unsigned long long now = global_ns();
        spent += counted_wait(last, now);
        last = now;
        if (spent > limit || *stop) return false;
    }
    return true;
}

// ---- one instance in one CTA: pointers, the state of a group's current ant
// and the pieces of a step

// KIND: how the ants take their steps and read a step's edge list (kShort, kLong,
// kTurns).
template <int L, int MODE, bool ALONE, int KIND>
struct Colony {
    static constexpr bool SPM = MODE != 0;
    static constexpr bool TURNS = KIND == kTurns;
    static_assert(!ALONE || KIND != kLong, "a CTA alone makes an index");
    static constexpr int V = 32 / L;
    static constexpr int NC = ALONE || TURNS ? 1 : kCopies;
    // Clusters: the vote on whether a wait gave up is taken with the one on the
    // list read behind it. On the matrix with 16 or 32 lanes it is taken at once,
    // which was faster there (ms per iteration at once and with the list's: n =
    // 1000, m = 256 2.66 and 2.77, m = 128 1.93 and 1.97; with eight lanes, 256
    // mixed instances, m = 64, 11.2 and 10.4).
    static constexpr bool VOTE_AT_ONCE = !ALONE && !SPM && L >= 16;
    using Entry = typename std::conditional<SPM, uint32_t, uint2>::type;   // edge key [, trail read]

    const ConstructArgs& A;
    const Group<L> G;
    int gl, lane, tid, nthr;
    int m, mp, C, rank, mc, a0, ml, ants_warps, s_slots;
    bool split;             // one ant per group: !TURNS (as a constant here, ptxas spills 13 registers more)
    // the instance
    int n, cl, W, Wp, dstrict;
    float tau0;
    bool write_all;
    uint32_t it, inst;
    const int2* xy;
    const uint2* rows;      // packed candidate rows
    const uint32_t* spos;
    const uint16_t* orders;
    const uint2* nodes;
    float* tau;             // matrix rows, or SPM values
    float* tauc;            // trails of the candidate rows
    uint32_t* tl;           // non-candidates with another trail
    int32_t* tl_cnt;
    int32_t* sidx;          // SPM only
    int32_t* stail;
    uint2* rec_g;
    uint32_t rec_words;
    int32_t* tours;
    int32_t* best;
    uint32_t* vis_base;
    // shared memory
    float* sP;
    uint32_t* s_cur;
    uint32_t* s_start;
    long long* s_len;
    Entry* elist;           // [kRing][mp]
    unsigned char* idx;     // the list's index
    int hshift;
    Misc* misc;
    int4* box;
    uint2* rec_s;
    int kbase;              // lists exchanged for earlier instances
    bool dead;              // a wait gave up (the same on a warp's lanes behind in_step())
    uint32_t n_fb, n_hit, n_miss;
    // the current ant
    uint32_t nv[V];         // candidates (or, on a fallback, the list of changed trails)
    float wv[V], tv[V];     // weights, trails
    uint32_t un;            // bit i: candidate i of this lane is unvisited
    uint32_t near;          // fallback: the nearest unvisited node (packed)
    int fb;                 // 0 candidates, 1 fallback, 2 fallback that must read every trail
    Order<L> order;         // the city's nearest boxes and number of listed trails (clusters:
    int changed;            // requested with the row, a fallback being in almost every step)
    uint32_t back;          // bit i: candidate i of this lane is the previous city
    Record<V> R;            // SPM: the current city's record

    __device__ __forceinline__ Colony(const ConstructArgs& a, bool sp)
        : A(a), G(threadIdx.x & 31), lane(threadIdx.x & 31), tid(threadIdx.x), nthr(blockDim.x), split(sp), kbase(0),
          dead(false)
    {
        gl = G.gl;
        m = A.m;
        mp = list_places(m);
        C = ALONE ? 1 : (int)cg::this_cluster().num_blocks();
        rank = ALONE ? 0 : (int)cg::this_cluster().block_rank();
        mc = A.mc;
        a0 = rank * mc;
        ml = max(0, min(m, a0 + mc) - a0);
        ants_warps = (ml * L + 31) >> 5;
        s_slots = A.s;
    }

    static __device__ __forceinline__ uint32_t key_of(const Entry& e)
    {
        if constexpr (SPM) return e;
        else return e.x;
    }
    __device__ __forceinline__ void sync_all() const
    {
        __syncwarp();
        if constexpr (ALONE) __syncthreads();
        else cg::this_cluster().sync();
    }
    // the CTA's warps that have ants meet (not in turns)
    __device__ __forceinline__ void ant_sync() const
    {
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"r"(ants_warps * 32) : "memory");
    }
    __device__ __forceinline__ uint2* rec_of(uint32_t r) const
    {
        if constexpr (MODE == 2 && ALONE) {
            return rec_s + r * rec_words;
        } else if constexpr (MODE == 2) {
            const uint32_t o = r % (uint32_t)C, li = r / (uint32_t)C;
            return cg::this_cluster().map_shared_rank(rec_s + li * rec_words, o);
        } else {
            return rec_g + (size_t)r * rec_words;
        }
    }
    // state that other SMs may have written (alone: this CTA's own stores)
    __device__ __forceinline__ float ld_f(const float* p) const { return ALONE ? *p : __ldcg(p); }
    __device__ __forceinline__ uint2 ld_rec(const uint2* p) const { return (ALONE || MODE == 2) ? *p : __ldcg(p); }
    __device__ __forceinline__ uint32_t pack(uint32_t id) const { return (__ldg(spos + id) << 16) | id; }
    __device__ __forceinline__ int slot(int k) const { return (kbase + k) & (kRing - 1); }
    // a list has mp places; those past m hold no edge
    __device__ __forceinline__ Entry* list(int k) const { return elist + slot(k) * mp; }
    // the matrix entry (u, v): u * n + v < 2^32
    __device__ __forceinline__ uint32_t at(uint32_t u, uint32_t v) const { return u * (uint32_t)n + v; }

    // Shared memory that does not depend on the instance; before any CTA pushes.
    __device__ __forceinline__ void open(unsigned char* smem)
    {
        const SmemLayout S = smem_layout(m, mc, A.nrec, s_slots, A.max_w, NC, TURNS, A.vis_in_smem,
                                         A.nodes_in_smem ? A.max_n : 0);
        sP = (float*)(smem + S.P);
        s_cur = (uint32_t*)(smem + S.cur);
        s_start = (uint32_t*)(smem + S.start);
        s_len = (long long*)(smem + S.len);
        elist = (Entry*)(smem + S.edges);
        idx = smem + S.index;
        hshift = 32 - index_bits(m);
        misc = (Misc*)(smem + S.misc);
        box = (int4*)(smem + S.box);
        rec_s = (uint2*)(smem + S.rec);
        vis_base = (uint32_t*)(smem + S.vis);
        nodes = (const uint2*)(smem + S.nodes);
        rec_words = (uint32_t)(s_slots + 1) * NC;
        uint32_t* e = (uint32_t*)elist;   // key 0 is no edge
#pragma unroll 1
        for (int i = tid; i < kRing * mp * (int)(sizeof(Entry) / 4); i += nthr) e[i] = 0u;
#pragma unroll 1
        for (int i = tid; i <= m; i += nthr) sP[i] = A.P[i];
        if constexpr (!ALONE) {
            if (tid == 0) {
                misc->stop = 0;
#pragma unroll 1
                for (int i = 0; i < kRing; ++i) {
                    // (hold, a test: an arrival that never comes for list 2)
                    const int h = i == 2 ? A.hold : kHoldNone;
                    mbar_init(smem_addr(&misc->bar[i]), 1 + (h == kHoldList));
                    mbar_init(smem_addr(&misc->sdone[i]), max(ants_warps, 1) + (h == kHoldStored));
                    mbar_init(smem_addr(&misc->pub[i]), C + (h == kHoldPublished));
                }
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
#pragma unroll 1
                for (int i = 0; i < kRing; ++i) mbar_expect(smem_addr(&misc->bar[i]), (uint32_t)(sizeof(Entry) * m));
            }
        }
    }

    // Instance b: pointers, tables, the SPM's working copies, every ant's first node.
    __device__ __forceinline__ void begin(int b)
    {
        const InstDesc D = A.desc[b];
        n = D.n;
        cl = D.cl;
        W = D.W;
        Wp = (W + 3) & ~3;
        dstrict = D.dstrict;
        tau0 = D.tau0;
        inst = (uint32_t)D.instance;
        xy = (const int2*)(A.xy) + D.xy_off;
        rows = A.rows + 32 * D.row_off;
        spos = A.spos + D.row_off;
        orders = A.order_boxes + (size_t)kOrder * D.row_off;
        const uint2* gnodes = A.snode + D.row_off;
        if (!A.nodes_in_smem) nodes = gnodes;
        tau = A.tau + D.tau_off;
        tauc = SPM ? nullptr : A.tauc + 32 * D.row_off;
        tl = SPM ? nullptr : A.tl_node + 32 * D.row_off;
        tl_cnt = SPM ? nullptr : A.tl_cnt + D.row_off;
        sidx = SPM ? A.spm_idx + D.tau_off : nullptr;
        stail = SPM ? A.spm_tail + D.node_off : nullptr;
        rec_g = SPM ? A.rec + (size_t)D.row_off * rec_words : nullptr;
        tours = A.tours + D.tour_off;
        best = A.best + D.node_off;
        write_all = !SPM && A.asym[b] != 0;
        if (!A.vis_in_smem) vis_base = A.vis_global + D.vis_off + (size_t)a0 * Wp;
        n_fb = n_hit = n_miss = 0u;

        if constexpr (SPM) {
            // working copies: copy 0 = the state at the start, written by "update 0"
            const int first = MODE == 2 ? rank + tid * C : rank * nthr + tid;
#pragma unroll 1
            for (int r = first; r < n; r += C * nthr) {
                uint2* X = rec_of(r);
#pragma unroll 1
                for (int q = 0; q < s_slots; ++q)
                    X[q * NC] = make_uint2((uint32_t)__ldcg(sidx + (size_t)r * s_slots + q),
                                           __float_as_uint(__ldcg(tau + (size_t)r * s_slots + q)));
                X[s_slots * NC] = make_uint2((uint32_t)__ldcg(stail + r), 0u);
                for (int i = 1; i < NC; ++i) X[s_slots * NC + i] = make_uint2(0u, 0xffffffffu);
            }
        }
        if (tid == 0) {
            misc->best_len = __ldcg(A.best_len + b);
            misc->iteration = __ldcg(A.iteration + b);
            for (int i = 0; i < 3; ++i) misc->stat[i] = 0ull;
        }
#pragma unroll 1
        for (int i = tid; i < W; i += nthr) box[i] = __ldg(A.box + D.word_off + i);
        if (A.nodes_in_smem) {
#pragma unroll 1
            for (int i = tid; i < n; i += nthr) const_cast<uint2*>(nodes)[i] = __ldg(gnodes + i);
        }
        if constexpr (TURNS) {   // heads of no list
#pragma unroll 1
            for (int i = tid; i < 2 << index_bits(m); i += nthr) ((uint32_t*)idx)[i] = 0u;
        }
        // visited words; the bits past the last node count as visited
#pragma unroll 1
        for (int i = tid; i < ml * Wp; i += nthr) {
            const int w = i % Wp;
            vis_base[i] = w < W - 1 ? 0u : w >= W ? 0xffffffffu : (n & 31) ? 0xffffffffu << (n & 31) : 0u;
        }
        __syncthreads();
        it = (uint32_t)misc->iteration;
        // step 0: first node of every ant (Alg. 1, uniform draw)
#pragma unroll 1
        for (int al = tid; al < ml; al += nthr) {
            const uint4 x = philox4x32_10(make_uint4(it, (uint32_t)(a0 + al), 0u, inst), A.key0, A.key1);
            const uint32_t start = pack(__umulhi(x.z, (uint32_t)n));
            s_cur[al] = start;
            s_start[al] = start;
            tours[(size_t)(a0 + al) * n] = (int)node_id(start);
            vis_base[(size_t)al * Wp + (start >> 21)] |= 1u << ((start >> 16) & 31);
        }
        sync_all();
    }

    // ---- staging of a city

    __device__ __forceinline__ void load_fallback(uint32_t ci)
    {
        order.load(orders + ci * (uint32_t)kOrder, gl);
        if constexpr (!SPM) changed = tl_cnt[ci];
    }
    __device__ __forceinline__ void load_city(uint32_t ci)
    {
        load_row<V>(rows + (ci * 32u + gl * V), nv, wv);
        if constexpr (!ALONE) load_fallback(ci);
    }
    __device__ __forceinline__ void load_cand_trails(uint32_t ci)
    {
        if constexpr (!SPM) load_trails<V>(tauc + (ci * 32u + gl * V), ALONE, tv);
    }
    // The visited bits of the row; `prev` = the city the ant came from. Sets fb
    // when every candidate is visited.
    __device__ __forceinline__ void check_row(uint32_t prev, const uint32_t* vis)
    {
        back = un = 0u;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const bool in = gl * V + i < cl;
            if (!SPM && in && node_id(nv[i]) == prev) back |= 1u << i;
            if (in && !visited(vis, nv[i] >> 16)) un |= 1u << i;
        }
        fb = G.ballot(un != 0u) ? 0 : 1;
    }
    // For the groups with `need` (every candidate visited): the nearest
    // unvisited node, and on the matrix the non-candidates whose trail is not
    // tau0 (fallback_trails() reads the trails).
    __device__ __forceinline__ void fallback(uint32_t c, const uint32_t* vis, bool need)
    {
        const uint32_t ci = node_id(c);
        const int2 pc = node_point(nodes[c >> 16]);
        if constexpr (ALONE) load_fallback(ci);
        if constexpr (!SPM) {
            if (need && changed > kChanged) fb = 2;
            if (need && fb == 1) {
                un = 0u;
                if (changed > 0) {
#pragma unroll
                    for (int i = 0; i < V; ++i) {
                        const int k = gl * V + i;
                        nv[i] = k < changed ? tl[ci * 32u + k] : 0u;
                        if (k < changed && !visited(vis, nv[i] >> 16)) un |= 1u << i;
                    }
                }
            }
            __syncwarp();
        }
        const bool search = need && fb == 1;
        const uint32_t to =
            nearest_unvisited<L>(G, order, pc, W, vis, nodes, box, spos, tau0, A.beta, dstrict, search);
        if (search) near = (min(to & 0xffffu, (uint32_t)n - 1u) << 16) | min(to >> 16, (uint32_t)n - 1u);
    }
    // trails of the listed non-candidates (matrix, fallback)
    __device__ __forceinline__ void fallback_trails(uint32_t ci, bool need)
    {
        if constexpr (!SPM) {
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (need && fb == 1 && ((un >> i) & 1u)) tv[i] = ld_f(tau + at(ci, node_id(nv[i])));
        }
    }
    // closing edge from city u to `start`: the trail in tv[0] of lane 0
    __device__ __forceinline__ void stage_closing(uint32_t u, uint32_t start)
    {
        if constexpr (!SPM) {
            fb = 1;
#pragma unroll
            for (int i = 0; i < V; ++i) nv[i] = gl == 0 && i == 0 ? start : 0xffffffffu;
            tv[0] = ld_f(tau + at(u, node_id(start)));
        }
    }

    // ---- a list's index (ants in turns, between barriers)
    //
    // Edges hang in chains by the hash of their key. A head holds (list << 11) |
    // ant, so that the heads of older lists are empty ones. Every ant then finds
    // the multiplicity of its edge in a chain of one or two entries, where reading
    // the list takes m / L loads a lane.
    //
    // SPM: the lowest ant's entry of every edge hangs by the hash of each end (entry
    // 2 j + side of ant j, the multiplicity in the upper half of its link), is
    // linked to the next ant's entry at the same city, and the first one's thread
    // replays the record's events in that order: a thread per record, where
    // groups of lanes that each replayed their ant's two records took 43,000
    // cycles a step at n = 100, m = 256.

    static constexpr uint32_t kEnd = 0xffffu;
    __device__ __forceinline__ uint32_t* edge_heads() const { return (uint32_t*)idx; }
    __device__ __forceinline__ uint32_t* city_heads() const { return edge_heads() + (1 << index_bits(m)); }
    __device__ __forceinline__ uint32_t* city_links() const { return city_heads() + (1 << index_bits(m)); }
    __device__ __forceinline__ uint16_t* edge_links() const { return (uint16_t*)(city_links() + 2 * mp); }
    __device__ __forceinline__ uint16_t* followers() const { return edge_links() + mp; }
    __device__ __forceinline__ uint32_t hash(uint32_t x) const { return (x * 2654435761u) >> hshift; }
    // the entry a head of list k holds, or kEnd
    static __device__ __forceinline__ uint32_t entry(uint32_t head, int k)
    {
        return (head >> 11) == (uint32_t)k ? head & 2047u : kEnd;
    }
    __device__ __forceinline__ uint32_t city_of(const Entry* E, uint32_t e) const
    {
        const uint32_t key = key_of(E[e >> 1]);
        return e & 1u ? key & 0xffffu : key >> 16;
    }
    // ant j's edge into list k's chains
    __device__ __forceinline__ void hang(int k, int j, uint32_t key) const
    {
        const uint32_t old = atomicExch(edge_heads() + hash(key), ((uint32_t)k << 11) | (uint32_t)j);
        edge_links()[j] = (uint16_t)entry(old, k);
    }
    // multiplicity of ant j's edge if j is the lowest ant on it, else 0
    __device__ __forceinline__ int lowest_on_edge(int k, int j) const
    {
        const Entry* E = list(k);
        const uint32_t mine = key_of(E[j]);
        int cnt = 0;
        bool lowest = true;
        uint32_t e = entry(edge_heads()[hash(mine)], k);
#pragma unroll 1
        while (e != kEnd) {
            const uint32_t key = key_of(E[e]), next = edge_links()[e];
            if (key == mine) {
                ++cnt;
                lowest = lowest && (int)e >= j;
            }
            e = next;
        }
        return lowest ? cnt : 0;
    }
    // Alg. 3 on a record in memory, by one thread
    __device__ __forceinline__ void replay(uint2* p, int& tail, uint32_t nb, float coef)
    {
        int hit = -1;
        float t = tau0;
#pragma unroll 4
        for (int q = 0; q < s_slots; ++q) {
            const uint2 x = ld_rec(p + q);
            if (x.x == nb) {
                hit = q;
                t = __uint_as_float(x.y);
            }
        }
        if (hit >= 0) {
            ++n_hit;
        } else {
            ++n_miss;
            if (A.skip_default) return;
            tail = tail + 1 == s_slots ? 0 : tail + 1;
            hit = tail;
        }
        p[hit] = make_uint2(nb, __float_as_uint(local_rule(t, tau0, coef)));
    }
    // SPM: the updates of list k, whose edges hang in their chains, on the records of
    // this CTA (record r belongs to CTA r mod C).
    __device__ __forceinline__ void update_records(int k)
    {
        if constexpr (SPM && TURNS) {
            const Entry* E = list(k);
            const uint32_t stamp = (uint32_t)k << 11;
            uint32_t* links = city_links();
#pragma unroll 1
            for (int j = tid; j < m; j += nthr) {
                const uint32_t cnt = (uint32_t)lowest_on_edge(k, j) << 16;
#pragma unroll
                for (uint32_t side = 0; side < 2; ++side) {
                    const uint32_t e = 2u * j + side, c = city_of(E, e);
                    uint32_t link = 0u;   // not listed: another ant's, or another CTA's record
                    if (cnt && (ALONE || c % (uint32_t)C == (uint32_t)rank))
                        link = cnt | entry(atomicExch(city_heads() + hash(c), stamp | e), k);
                    links[e] = link;
                }
            }
            __syncthreads();
            uint32_t firsts = 0u;   // bit i: this thread's i-th entry is its city's first (2 m <= 32 nthr)
#pragma unroll 1
            for (int i = 0, e = tid; e < 2 * m; ++i, e += nthr) {
                if (!(links[e] >> 16)) continue;
                const uint32_t c = city_of(E, e);
                bool first = true;
                uint32_t next = kEnd;
                uint32_t x = entry(city_heads()[hash(c)], k);
#pragma unroll 1
                while (x != kEnd) {
                    const uint32_t xc = city_of(E, x), link = links[x];
                    if (xc == c) {
                        first = first && x >= (uint32_t)e;
                        if (x > (uint32_t)e) next = min(next, x);
                    }
                    x = link & 0xffffu;
                }
                followers()[e] = (uint16_t)next;
                if (first) firsts |= 1u << i;
            }
            __syncthreads();
#pragma unroll 1
            for (int i = 0, e0 = tid; e0 < 2 * m; ++i, e0 += nthr) {
                if (!((firsts >> i) & 1u)) continue;
                const uint32_t c = city_of(E, e0);
                uint2* p = rec_of(c);
                int tail = (int)ld_rec(p + s_slots).x;
                uint32_t e = (uint32_t)e0;
#pragma unroll 1
                do {
                    replay(p, tail, other_end(key_of(E[e >> 1]), c), sP[links[e] >> 16]);
                    e = followers()[e];
                } while (e != kEnd);
                p[s_slots] = make_uint2((uint32_t)tail, (uint32_t)k);
            }
        }
    }

    // ---- edge lists

    // Entries are read four per lane at a time; a short list is read at once.
    __device__ __forceinline__ int list_end() const { return KIND == kShort ? 1 : m; }

    // Multiplicity of edge `key` in list k and the lowest ant that took it.
    __device__ __forceinline__ int count(int k, uint32_t key, int& low) const
    {
        const Entry* E = list(k);
        uint32_t cnt = 0u, lo = 0xffffffffu;
#pragma unroll 1
        for (int j0 = 0; j0 < list_end(); j0 += 4 * L) {
#pragma unroll
            for (int i = 3; i >= 0; --i) {
                const int x = j0 + i * L + gl;
                const bool is = key_of(E[x]) == key;   // (places past the list hold no edge)
                cnt += is ? 1u : 0u;
                lo = is ? min(lo, (uint32_t)x) : lo;
            }
        }
        low = (int)G.min_u32(lo);
        return (int)G.add_u32(cnt);
    }
    // Multiplicity of ant a's edge and the lowest ant that took it (or -1 where
    // that is another). With many more ants than cities the chains are longer than a
    // lane's share of the list (16 CTAs, n = 50, m = 1024: 0.6 ms an
    // iteration by chain, 0.33 by list; 200 of n = 100, m = 256: 2.11 and 2.03).
    __device__ __forceinline__ int own_edge(int k, int a, bool on, int& low) const
    {
        if (!TURNS || 2 * m >= 3 * n) return count(k, key_of(list(k)[a]), low);
        const int cnt = on ? lowest_on_edge(k, a) : 0;
        low = cnt > 0 ? a : -1;
        __syncwarp();
        return cnt;
    }
    // Four entries of a list per lane, 4 L in all from entry j0 on (keys k0 ..
    // k3), and which of them touch city c: bit l of h_i = entry j0 + i L + l.
    // (Scalars: an array indexed at run time would live in local memory.)
    struct Part {
        uint32_t k0, k1, k2, k3;
        unsigned h0, h1, h2, h3;
        __device__ __forceinline__ bool some() const { return (h0 | h1 | h2 | h3) != 0u; }
        // the first entry left, taken out; -1: none
        __device__ __forceinline__ int take()
        {
            if (h0) {
                const int at = __ffs(h0) - 1;
                h0 &= h0 - 1u;
                return at;
            }
            if (h1) {
                const int at = L + __ffs(h1) - 1;
                h1 &= h1 - 1u;
                return at;
            }
            if (h2) {
                const int at = 2 * L + __ffs(h2) - 1;
                h2 &= h2 - 1u;
                return at;
            }
            if (!h3) return -1;
            const int at = 3 * L + __ffs(h3) - 1;
            h3 &= h3 - 1u;
            return at;
        }
    };
    // The entries from j0 on, and whether any but ant a's touches city c or is
    // the edge `mine`, for this lane.
    __device__ __forceinline__ bool read_part(const Entry* E, int j0, uint32_t c, uint32_t mine, int a, Part& P) const
    {
        const int j = j0 + gl, skip = a - j;
        P.k0 = key_of(E[j]);
        P.k1 = key_of(E[j + L]);
        P.k2 = key_of(E[j + 2 * L]);
        P.k3 = key_of(E[j + 3 * L]);
        const auto is = [&](uint32_t key, int i) {
            return (touches(key, c) || (ALONE && !SPM && key == mine)) && skip != i * L;
        };
        const bool b0 = is(P.k0, 0), b1 = is(P.k1, 1), b2 = is(P.k2, 2), b3 = is(P.k3, 3);
        P.h0 = b0;
        P.h1 = b1;
        P.h2 = b2;
        P.h3 = b3;
        return b0 || b1 || b2 || b3;
    }
    // ... and which lanes hold one, for the groups with `on`
    __device__ __forceinline__ void vote_part(bool on, Part& P) const
    {
        P.h0 = G.ballot(on && P.h0);
        P.h1 = G.ballot(on && P.h1);
        P.h2 = G.ballot(on && P.h2);
        P.h3 = G.ballot(on && P.h3);
    }
    // matrix: brings the trails of the candidates (or listed nodes) of city ci
    // up to list k. The list's edges at ci are gone through in ant order: the
    // lowest ant's trail of an edge counts, and how many took it. a >= 0: the
    // ant's own edge `mine` is in the list; its multiplicity and lowest ant come
    // back (its trail is not set: where the ant came from is visited). A CTA
    // alone asks for these only: its trails are read behind the updates.
    __device__ __forceinline__ void overlay(int k, uint32_t ci, uint32_t mine, int a, bool on, int& kown, int& low)
    {
        kown = 1;
        low = a;
        if constexpr (!SPM) {
            const Entry* E = list(k);
            int cnt[V];
            float t_low[V];
#pragma unroll
            for (int i = 0; i < V; ++i) {
                cnt[i] = 0;
                t_low[i] = tau0;
            }
            bool some = false;
#pragma unroll 1
            for (int j0 = 0; j0 < list_end(); j0 += 4 * L) {
                Part P;
                const bool has = read_part(E, j0, ci, mine, a, P);
                if (!any_lane((on && has) || (!VOTE_AT_ONCE && dead))) continue;   // usual: nobody else at this city
                if (!ALONE && !VOTE_AT_ONCE && !in_step()) return;
                vote_part(on, P);
                some = true;
#pragma unroll 1
                while (G.any_group(P.some())) {
                    const int to = P.take();
                    const Entry x = E[j0 + max(to, 0)];
                    const uint32_t o = to < 0 ? kNoCity : other_end(x.x, ci);
                    if (to >= 0 && x.x == mine) {
                        ++kown;
                        low = min(low, j0 + to);
                    }
                    if constexpr (!ALONE) {
#pragma unroll
                        for (int i = 0; i < V; ++i)
                            if (node_id(nv[i]) == o) {
                                t_low[i] = cnt[i] == 0 ? __uint_as_float(x.y) : t_low[i];
                                ++cnt[i];
                            }
                    }
                }
            }
            if (!ALONE && some) {
#pragma unroll
                for (int i = 0; i < V; ++i)
                    if (cnt[i] > 0) tv[i] = local_rule(t_low[i], tau0, sP[cnt[i]]);
            }
        }
    }

    // ---- SPM records

    __device__ __forceinline__ void load_record(uint32_t r, uint2 (&raw)[NC][V], uint2 (&meta)[NC]) const
    {
        const uint2* p = rec_of(r);
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int q = i * L + gl;
#pragma unroll
            for (int c = 0; c < NC; ++c)
                raw[c][i] = q < s_slots ? ld_rec(p + q * NC + c) : make_uint2(0xffffffffu, 0u);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) meta[c] = ld_rec(p + s_slots * NC + c);
    }
    // the latest copy written by update `lim` or before
    static __device__ __forceinline__ void pick_copy(const uint2 (&raw)[NC][V], const uint2 (&meta)[NC], int lim,
                                                     Record<V>& X)
    {
        X.buf = 0;
        int tag = (int)meta[0].y;
        if (NC > 1 && tag > lim) tag = -2;
        X.tail = (int)meta[0].x;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            X.idx[i] = (int32_t)raw[0][i].x;
            X.val[i] = __uint_as_float(raw[0][i].y);
        }
#pragma unroll
        for (int c = 1; c < NC; ++c) {
            const int t = (int)meta[c].y;
            const bool take = t <= lim && t > tag;
            tag = take ? t : tag;
            X.buf = take ? c : X.buf;
            X.tail = take ? (int)meta[c].x : X.tail;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                X.idx[i] = take ? (int32_t)raw[c][i].x : X.idx[i];
                X.val[i] = take ? __uint_as_float(raw[c][i].y) : X.val[i];
            }
        }
    }
    __device__ __forceinline__ void read_record(uint32_t r, int lim, Record<V>& X) const
    {
        if constexpr (SPM) {
            uint2 raw[NC][V], meta[NC];
            load_record(r, raw, meta);
            pick_copy(raw, meta, lim, X);
        }
    }
    // Alg. 3 on the private copy: a hit updates in place (the highest slot that
    // holds nb), a miss evicts the slot after the tail
    __device__ __forceinline__ bool apply_event(Record<V>& X, uint32_t nb, float coef, bool on) const
    {
        int hit = -1;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const unsigned q = G.ballot(X.idx[i] == (int32_t)nb);   // lanes past the slots hold -1
            if (q) hit = i * L + 31 - __clz(q);
        }
        int put = hit;
        if (!on) {
            put = -1;
        } else if (hit < 0 && !A.skip_default) {
            X.tail = X.tail + 1 == s_slots ? 0 : X.tail + 1;
            put = X.tail;
        }
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (i * L + gl == put) {
                X.idx[i] = (int32_t)nb;
                X.val[i] = local_rule(hit >= 0 ? X.val[i] : tau0, tau0, coef);
            }
        return hit >= 0;
    }
    __device__ __forceinline__ void store_record(uint32_t r, const Record<V>& X, int tag) const
    {
        uint2* p = rec_of(r) + X.buf;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const int q = i * L + gl;
            if (q < s_slots) p[q * NC] = make_uint2((uint32_t)X.idx[i], __float_as_uint(X.val[i]));
        }
        if (gl == 0) p[s_slots * NC] = make_uint2((uint32_t)X.tail, (uint32_t)tag);
    }
    // The events of list k on record r, in the order of the lowest ant of each
    // distinct edge, for the groups with `on`. True if ant a is the lowest that
    // touches r: it counted them and has to store X (with `store_only` nobody
    // else needs X). nb: the other end of ant a's edge when it touches r, kNoCity
    // when it does not.
    __device__ __forceinline__ bool events(int k, uint32_t r, Record<V>& X, int a, uint32_t nb, bool store_only,
                                           bool on)
    {
        if constexpr (SPM) {
            const Entry* E = list(k);
            int first = -1;
            uint32_t hits = 0u, ev = 0u;
            const bool own = nb != kNoCity;   // E[a] touches r
            bool go_on = on, others = false;
#pragma unroll 1
            for (int j0 = 0; j0 < list_end(); j0 += 4 * L) {
                Part P;
                others |= read_part(E, j0, r, kNoEdge, own ? a : -1, P);
            }
            if (!any_lane((on && others) || dead)) {
                // usual: at most the ant's own edge
                const bool one = on && own;
                if (G.any_group(one)) hits = apply_event(X, nb, sP[1], one) && one ? 1u : 0u;
                if (one) {
                    first = a;
                    ev = 1u;
                }
            } else {
                if (!ALONE && !in_step()) return false;
#pragma unroll 1
                for (int j0 = 0; j0 < list_end(); j0 += 4 * L) {
                    Part P;
                    read_part(E, j0, r, kNoEdge, -1, P);
                    vote_part(go_on, P);
#pragma unroll 1
                    while (G.any_group(P.some())) {
                        const int to = P.take();
                        if (to >= 0 && first < 0) {
                            first = j0 + to;
                            if (store_only && first != a) {
                                go_on = false;
                                P.h0 = P.h1 = P.h2 = P.h3 = 0u;
                            }
                        }
                        const uint32_t key = key_of(E[j0 + max(to, 0)]);
                        int lo, cnt;
                        if constexpr (KIND == kShort) {
                            // the whole list is in registers; the edge's other
                            // entries are done with
                            const unsigned q0 = G.ballot(P.k0 == key), q1 = G.ballot(P.k1 == key);
                            const unsigned q2 = G.ballot(P.k2 == key), q3 = G.ballot(P.k3 == key);
                            cnt = __popc(q0) + __popc(q1) + __popc(q2) + __popc(q3);
                            P.h0 &= ~q0;
                            P.h1 &= ~q1;
                            P.h2 &= ~q2;
                            P.h3 &= ~q3;
                            lo = to;
                        } else {
                            cnt = count(k, key, lo);
                        }
                        const bool go = go_on && to >= 0 && lo == j0 + to;
                        const bool hit = apply_event(X, other_end(key, r), sP[min(cnt, m)], go);
                        if (go) {
                            ++ev;
                            hits += hit ? 1u : 0u;
                        }
                    }
                }
            }
            // the update goes to the copy after the latest (one copy: in place)
            if (NC > 1 && split && first >= 0) X.buf = X.buf + 1 == NC ? 0 : X.buf + 1;
            const bool mine = first >= 0 && first == a;
            if (mine && gl == 0) {
                n_hit += hits;
                n_miss += ev - hits;
            }
            return mine;
        }
        return false;
    }
    // trails of the candidates from the record (absent: tau0; the highest slot
    // that holds a node counts)
    __device__ __forceinline__ void match(const Record<V>& X)
    {
        if constexpr (SPM) {
#pragma unroll
            for (int i = 0; i < V; ++i) tv[i] = tau0;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                constexpr int B = L < 8 ? L : 8;
#pragma unroll 1
                for (int q0 = 0; q0 < L && i * L + q0 < s_slots; q0 += B) {
#pragma unroll
                    for (int q = 0; q < B; ++q) {
                        const int32_t id = G.shfl(X.idx[i], q0 + q);
                        const float t = G.shfl(X.val[i], q0 + q);
#pragma unroll
                        for (int v = 0; v < V; ++v)
                            if ((int32_t)node_id(nv[v]) == id) tv[v] = t;
                    }
                }
            }
        }
    }

    // ---- selection

    // Alg. 2 when the row's every trail has to be read (fb == 2), behind the
    // publication of the updates before list `pending`'s (0: none). Those of
    // `pending` may not be published: the lowest ant's trail and the edge's
    // multiplicity give the updated trail.
    __device__ __forceinline__ void read_all(uint32_t ci, int2 pc, const uint32_t* vis, int pending,
                                             unsigned long long& key, float& tk) const
    {
        if constexpr (!SPM) {
#pragma unroll 1
            for (int j = gl; j < n; j += L) {
                if (visited(vis, __ldg(spos + j))) continue;
                float t = ld_f(tau + at(ci, (uint32_t)j));
                if (pending > 0) {
                    const Entry* E = list(pending);
                    const uint32_t key = edge_key(ci, (uint32_t)j);
                    int cnt = 0, lo = 0;
#pragma unroll 1
                    for (int q = m - 1; q >= 0; --q)
                        if (E[q].x == key) {
                            ++cnt;
                            lo = q;
                        }
                    if (cnt) t = local_rule(__uint_as_float(E[lo].y), tau0, sP[cnt]);
                }
                const unsigned long long k2 =
                    pack_pj(__fmul_rn(t, heuristic(euc2d(pc, __ldg(xy + j)), A.beta)), j);
                if (k2 > key) {
                    key = k2;
                    tk = t;
                }
            }
        }
    }

    // Eq. 1, Eq. 2 or Alg. 2's full scan for the groups with `on`: the next
    // city (packed) and the trail of the edge taken. pending > 0: the updates of
    // that list may not be published (clusters, one ant per group).
    __device__ __forceinline__ uint32_t select(uint32_t c, const uint32_t* vis, float u_q, float u_r, int pending,
                                               bool on, float& t_edge)
    {
        const bool cand = on && fb == 0;
        uint32_t nx = c;
        if (G.any_group(cand)) {
            float v[V];
#pragma unroll
            for (int i = 0; i < V; ++i) v[i] = (un >> i) & 1u ? __fmul_rn(tv[i], wv[i]) : 0.0f;
            const bool explore = cand && !(u_q < A.q0);
            // exploitation: argmax of tau*eta^beta, ties -> lowest rank.
            // Non-negative floats order like their bit patterns.
            uint32_t mb = 0u;
#pragma unroll
            for (int i = 0; i < V; ++i) mb = max(mb, __float_as_uint(v[i]));   // 0 where visited
            mb = G.max_u32(mb);
            int mine = 0;   // this lane's candidate, if its lane is chosen
            bool has = false;
#pragma unroll
            for (int i = V - 1; i >= 0; --i)
                if (((un >> i) & 1u) && __float_as_uint(v[i]) == mb) {
                    mine = i;
                    has = true;
                }
            const unsigned bx = G.ballot(has);
            int src = bx ? __ffs(bx) - 1 : 0;
            if (G.any_group(explore)) {
                // exploration: roulette of Eq. 2 over a 32-position inclusive
                // Hillis-Steele scan (offsets 1,2,4,8,16)
                float P[V];
#pragma unroll
                for (int i = 0; i < V; ++i) P[i] = v[i];
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    float y[V];
                    if (off >= V) {
                        const int dl = off / V;
#pragma unroll
                        for (int i = 0; i < V; ++i) {
                            const float o = G.shfl_up(P[i], dl);
                            y[i] = gl >= dl ? __fadd_rn(P[i], o) : P[i];
                        }
                    } else {
                        float prev[V];
#pragma unroll
                        for (int i = 0; i < V; ++i) {
                            // positions i < off read the previous lane's V-off+i
                            if (i < off) prev[i] = G.shfl_up(P[i - off + V], 1);
                        }
#pragma unroll
                        for (int i = 0; i < V; ++i) {
                            if (i >= off) y[i] = __fadd_rn(P[i], P[i - off]);
                            else y[i] = gl >= 1 ? __fadd_rn(P[i], prev[i]) : P[i];
                        }
                    }
#pragma unroll
                    for (int i = 0; i < V; ++i) P[i] = y[i];
                }
                const float t = __fmul_rn(u_r, G.shfl(P[V - 1], L - 1));
                int first = -1, last = -1, firstu = -1;
#pragma unroll
                for (int i = 0; i < V; ++i) {
                    const bool u = (un >> i) & 1u, pos = u && v[i] > 0.0f;
                    if (first < 0 && pos && P[i] > t) first = i;
                    if (pos) last = i;
                    if (firstu < 0 && u) firstu = i;
                }
                const unsigned bf = G.ballot(first >= 0);
                const unsigned bl = G.ballot(last >= 0);
                const unsigned bu = G.ballot(firstu >= 0);
                if (explore) {
                    src = bf ? __ffs(bf) - 1 : bl ? 31 - __clz(bl) : bu ? __ffs(bu) - 1 : 0;
                    mine = bf ? first : bl ? last : firstu;
                }
            }
            uint32_t myn = nv[0];
            float myt = tv[0];
#pragma unroll
            for (int i = 1; i < V; ++i)
                if (mine == i) {
                    myn = nv[i];
                    myt = tv[i];
                }
            if constexpr (!SPM) t_edge = G.shfl(myt, src);
            nx = G.shfl(myn, src);
        }
        const bool scan = on && fb != 0;
        if (!G.any_group(scan)) return nx;

        // Alg. 2: the largest product over all unvisited nodes, ties -> lowest node
        if (scan && gl == 0) ++n_fb;
        const uint32_t ci = node_id(c);
        // nodes whose trail is not tau0, if any is unvisited
        uint32_t open = 0u;
        if (scan && fb == 1) {
            if constexpr (SPM) {
#pragma unroll
                for (int i = 0; i < V; ++i)
                    if (R.idx[i] >= 0 && !visited(vis, __ldg(spos + R.idx[i]))) open |= 1u << i;
            } else {
                open = un;
            }
        }
        const unsigned opened = G.ballot(open != 0u);   // (by the whole warp)
        const bool weigh = scan && (fb == 2 || opened != 0u);
        if (scan) {
            nx = near;
            t_edge = tau0;
        }
        if (!G.any_group(weigh)) return nx;
        const int2 pc = __ldg(xy + ci);
        unsigned long long key = 0ull;
        float tk = tau0;   // the trail behind this lane's key
        if (weigh && fb == 1) {
#pragma unroll
            for (int i = 0; i <= V; ++i) {
                // i == V: the nearest node, on lane 0. A changed trail is never
                // below tau0, so on equal keys of one node it is the node's.
                const bool here = i < V ? (open >> i) & 1u : gl == 0;
                if (!here) continue;
                const int j = i < V ? (SPM ? R.idx[i < V ? i : 0] : (int)node_id(nv[i < V ? i : 0])) : (int)node_id(near);
                const float t = i < V ? (SPM ? R.val[i < V ? i : 0] : tv[i < V ? i : 0]) : tau0;
                const unsigned long long k2 =
                    pack_pj(__fmul_rn(t, heuristic(euc2d(pc, __ldg(xy + j)), A.beta)), j);
                if (k2 > key) {
                    key = k2;
                    tk = t;
                }
            }
        }
        __syncwarp();
        if constexpr (!SPM && !ALONE) {
            // read_all() needs every update before list `pending`'s; the wait of
            // the staging was for those before the list ahead of it. (Every ant
            // stores them before it waits for the list after `pending`.)
            if (pending > 1 && any_lane(weigh && fb == 2)) {
                wait_bar(misc->pub, pending - 1);
                if (!in_step()) return nx;
            }
        }
        if (weigh && fb == 2) read_all(ci, pc, vis, pending, key, tk);
        __syncwarp();
        const unsigned long long kmax = G.max_key(key);
        uint32_t id = 0xffffffffu - (uint32_t)(kmax & 0xffffffffull);
        // lanes that hold the same key hold the same node: its listed trail, if
        // any lane has one, is the one that changed
        const unsigned same = G.ballot(key == kmax && tk != tau0);
        const float ts = G.shfl(tk, same ? __ffs(same) - 1 : 0);
        if (weigh) {
            if (kmax == 0ull || id >= (uint32_t)n) {
                // no unvisited node: cannot happen before step n
                if (gl == 0) atomicExch(A.status, 4);
                id = ci;
            }
            nx = pack(id);
            if (!SPM && same) t_edge = ts;
        }
        return nx;
    }

    // ---- matrix updates

    // The updated trail of edge (u, v) in both halves and in the candidate
    // rows; bu, bv: bit i = candidate i of this lane in u's row is v, in v's
    // row u. An unchanged trail (tau0 on most edges early on) is not stored.
    __device__ __forceinline__ void store_edge(uint32_t u, uint32_t v, float t_old, float t2, uint32_t bu,
                                               uint32_t bv) const
    {
        if constexpr (!SPM) {
            if (__float_as_uint(t_old) == __float_as_uint(t2) && !write_all) return;
            if (gl < 2) tau[gl ? at(v, u) : at(u, v)] = t2;
#pragma unroll
            for (int i = 0; i < V; ++i) {
                if ((bu >> i) & 1u) tauc[u * 32u + gl * V + i] = t2;
                if ((bv >> i) & 1u) tauc[v * 32u + gl * V + i] = t2;
            }
        }
    }
    // the update of ant a's edge (u, v) from the list alone: the closing edges,
    // and the steps of a CTA with more ants than groups
    __device__ __forceinline__ void fold_edge(int list_no, int a, uint32_t u, uint32_t v, bool on) const
    {
        if constexpr (!SPM) {
            const Entry* E = list(list_no);
            int low;
            const int k = own_edge(list_no, a, on, low);
            if (!on || low != a) return;   // (no collective follows)
            const float t = __uint_as_float(E[a].y);
            uint32_t bits[2];
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                uint32_t ids[V];
                float w[V];
                load_row<V>(rows + ((side ? v : u) * 32u + gl * V), ids, w);
                bits[side] = 0u;
#pragma unroll
                for (int i = 0; i < V; ++i)
                    if (gl * V + i < cl && node_id(ids[i]) == (side ? u : v)) bits[side] |= 1u << i;
            }
            store_edge(u, v, t, local_rule(t, tau0, sP[k]), bits[0], bits[1]);
        }
    }

    // Waits for list k's barrier in the ring `bars`, by the whole warp. A lane
    // whose wait gave up goes on without the data until in_step().
    __device__ __forceinline__ void wait_bar(unsigned long long* bars, int k)
    {
        const int kk = kbase + k;
        const uint32_t bar = smem_addr(&bars[kk & (kRing - 1)]), parity = (uint32_t)((kk - 1) / kRing) & 1u;
        if (!mbar_test(bar, parity) && (dead || !mbar_wait(bar, parity, A.wait_ns, &misc->stop))) dead = true;
    }
    // False, on all lanes, when a wait of the warp gave up: the status is raised,
    // the cluster's other waits are told, and the warp must leave for finish(). It
    // has formed no index and stored nothing from data that did not come, and
    // reads and sends nothing more.
    __device__ __forceinline__ bool in_step()
    {
        if (__all_sync(0xffffffffu, !dead)) return true;
        dead = true;
        if (lane == 0) atomicExch(A.status, kWaitGaveUp);
        if (lane < C) *cg::this_cluster().map_shared_rank(&misc->stop, lane) = 1;
        __syncwarp();
        return false;
    }

    // The publisher warp of a cluster's CTA (one ant per group).
    __device__ __forceinline__ void publish()
    {
#pragma unroll 1
        for (int k = 1; k <= n / A.period; ++k) {
            wait_bar(misc->bar, k);
            if (!in_step()) return;
            // ready for list k + kRing, which nobody sends before this CTA's
            // ants have pushed list k + kRing - 1
            if (lane == 0) mbar_expect(smem_addr(&misc->bar[slot(k)]), (uint32_t)(sizeof(Entry) * m));
            if (ml > 0) wait_bar(misc->sdone, k);
            if (!in_step()) return;
            if (lane < C) mbar_arrive_remote(remote_addr(smem_addr(&misc->pub[slot(k)]), lane));
        }
    }

    // One ant per group: its whole tour. Groups without an ant go along.
    __device__ __forceinline__ void walk()
    {
        const int group = tid / L;
        const bool act = group < ml;
        const int al = act ? group : 0, a = a0 + al;
        uint32_t* vis = vis_base + (size_t)al * Wp;
        const uint32_t start = s_start[al];
        uint32_t c = start;
        int32_t* tour = tours + (size_t)a * n;
        int tb = (int)node_id(c);   // the tour's last L nodes, one per lane
        uint32_t qx = 0u, qy = 0u;  // the draws of L steps, one per lane
        float u_q = 0.0f, u_r = 0.0f;
        int k = 0;                  // lists that are complete
        int left = A.period;        // steps to the next update
        // cluster addresses of this lane's receiver (when one lane serves each CTA)
        const bool one_each = !ALONE && L >= C;
        const uint32_t far_list = one_each ? remote_addr(smem_addr(elist), min(gl, C - 1)) : 0u;
        const uint32_t far_bar = one_each ? remote_addr(smem_addr(misc->bar), min(gl, C - 1)) : 0u;
        // the last update, stored behind the next push: (pu, pv) the edge;
        // matrix: old and new trail and its places in the candidate rows; SPM:
        // the record of pu before it
        uint32_t pu = 0u, pv = 0u, pbu = 0u, pbv = 0u;
        float pt = 0.0f, pt2 = 0.0f;
        bool pstore = false;        // matrix: store the trail; SPM: store record pv
        bool owed = false;          // list k's update is not stored yet
        Record<V> U;
        // Step 0 stages the first city only; step n pushes the closing edge.
#pragma unroll 1
        for (int step = 0; step <= n; ++step) {
            const uint32_t u = node_id(c);
            uint32_t v = u, key = 0u, bu = 0u;
            float t_edge = tau0;
            const bool upd = step > 0 && --left == 0;
            if (upd) left = A.period;
            if (step > 0) {
                uint32_t nx = start;
                if (step < n) nx = select(c, vis, u_q, u_r, ALONE ? 0 : k, act, t_edge);
                else if constexpr (!SPM) t_edge = G.shfl(tv[0], 0);
                if constexpr (!SPM && !ALONE) {
                    if (dead) return;
                }
                v = node_id(nx);
                key = edge_key(u, v);
                if (upd) {
                    Entry x;
                    if constexpr (SPM) x = key;
                    else x = make_uint2(key, __float_as_uint(t_edge));
                    const uint32_t eo = (uint32_t)(slot(k + 1) * mp + a) * (uint32_t)sizeof(Entry);
                    if constexpr (ALONE) {
                        if (act && gl == 0) list(k + 1)[a] = x;
                    } else if (L >= C) {
                        if (act && gl < C) st_async(far_list + eo, far_bar + 8u * slot(k + 1), x);
                    } else {
#pragma unroll 1
                        for (int r = gl; act && r < C; r += L)
                            st_async(remote_addr(smem_addr(elist) + eo, r),
                                     remote_addr(smem_addr(&misc->bar[slot(k + 1)]), r), x);
                    }
                }
                c = nx;
                if constexpr (!SPM) {
#pragma unroll
                    for (int i = 0; i < V; ++i)
                        if (fb == 0 && gl * V + i < cl && node_id(nv[i]) == v) bu |= 1u << i;
                }
            }
            if (step < n) {
                const int sl = step & (L - 1);
                load_city(v);
                if (act && gl == 0 && step > 0) vis[c >> 21] |= 1u << ((c >> 16) & 31);
                if (gl == sl) tb = (int)v;
                if (act && sl == L - 1) tour[step - sl + gl] = tb;
            }
            uint2 raw[NC][V], meta[NC];
            if constexpr (!ALONE) {
                __syncwarp();
                if (k > 1) wait_bar(misc->pub, k - 1);   // usually long complete
                if (VOTE_AT_ONCE && k > 1 && !in_step()) return;
            }
            if constexpr (SPM) load_record(v, raw, meta);
            else if (!ALONE && step < n) load_cand_trails(v);
            if constexpr (!ALONE) {
                if (owed) {
                    settle(k, pu, pv, U, a, pstore, pt, pt2, pbu, pbv, act);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_addr(&misc->sdone[slot(k)]));
                    owed = false;
                }
            }
            Record<V> X;   // SPM: the next city's record
            __syncwarp();
            if (step < n) {
                const int s1 = (step + 1) & (L - 1);
                if (s1 == 0 || step == 0) {   // the draws of steps step + 1 ..
                    const uint4 x = philox4x32_10(
                        make_uint4(it, (uint32_t)a, (uint32_t)(step + 1 - s1 + gl), inst), A.key0, A.key1);
                    qx = x.x;
                    qy = x.y;
                }
                u_q = unit24(G.shfl(qx, s1));
                u_r = unit24(G.shfl(qy, s1));
                check_row(step > 0 ? u : kNoCity, vis);
                if (step + 1 < n) {
                    const bool need = act && fb != 0;
                    if (G.any_group(need)) {
                        fallback(c, vis, need);
                        if constexpr (!ALONE) fallback_trails(v, need);
                    }
                } else if constexpr (!ALONE) {
                    stage_closing(v, start);
                }
                if constexpr (!SPM && !ALONE) {
                    int d0, d1;
                    if (k > 0) overlay(k, v, kNoEdge, -1, act, d0, d1);
                }
            }
            if constexpr (SPM) {
                pick_copy(raw, meta, max(k - 1, 0), X);
                if (!ALONE && k > 0) events(k, v, X, -1, kNoCity, false, act);
            }
            if (upd) {
                if constexpr (ALONE) {
                    ant_sync();   // the list is complete
                } else {
                    wait_bar(misc->bar, k + 1);
                    if (VOTE_AT_ONCE && !in_step()) return;
                    // the closing edge's trail is stored at once (fold_edge()), and
                    // the ants of other CTAs may still be storing list k's, one of
                    // which can be the same edge's: theirs first. (They do so before
                    // they wait for list k + 1; once an iteration.)
                    if (!SPM && step == n) {
                        if (k > 0) wait_bar(misc->pub, k);
                        if (!in_step()) return;
                    }
                }
                ++k;
                owed = true;
                pu = u;
                pv = v;
                pstore = false;
                if constexpr (SPM) {
                    U = R;
                    pstore = events(k, v, X, a, u, false, act);
                } else if (step == n) {
                    fold_edge(k, a, u, v, act);
                } else {
                    int ko, low;
                    // alone, every trail is read when the updates are stored
                    overlay(k, ALONE ? kNoCity : v, key, a, act, ko, low);
                    pstore = low == a;
                    pt = t_edge;
                    pt2 = local_rule(t_edge, tau0, sP[min(ko, m)]);
                    pbu = bu;
                    pbv = back;
                }
                if constexpr (!ALONE && !VOTE_AT_ONCE) {
                    if (dead) return;   // (voted on while the list was read)
                }
            } else if constexpr (!ALONE && !VOTE_AT_ONCE) {
                if (A.period > 1 && !in_step()) return;   // (the wait for publication)
            }
            if constexpr (SPM) {
                R = X;
                match(R);
            }
            if (owed && (ALONE || step == n)) {
                settle(k, pu, pv, U, a, pstore, pt, pt2, pbu, pbv, act);
                if constexpr (ALONE) {
                    ant_sync();   // its updates are stored
                } else {
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_addr(&misc->sdone[slot(k)]));
                }
                owed = false;
            }
            if constexpr (ALONE && !SPM) {
                if (step < n) {
                    if (step + 1 == n) {
                        stage_closing(v, start);
                    } else {
                        if (fb == 0) load_cand_trails(v);
                        fallback_trails(v, act && fb == 1);
                    }
                }
            }
        }
        const int last = (n - 1) & (L - 1);
        if (act && last != L - 1 && gl <= last) tour[n - 1 - last + gl] = tb;
    }
    // stores the update of list k that belongs to ant a (see walk())
    __device__ __forceinline__ void settle(int k, uint32_t pu, uint32_t pv, Record<V>& U, int a, bool pstore, float pt,
                                           float pt2, uint32_t pbu, uint32_t pbv, bool act)
    {
        if constexpr (SPM) {
            if (events(k, pu, U, a, pv, true, act)) store_record(pu, U, k);
            if (pstore) store_record(pv, R, k);
        } else {
            if (act && pstore) store_edge(pu, pv, pt, pt2, pbu, pbv);
        }
    }

    // In turns: every read is between two full barriers, and a group takes several
    // ants when there are more of them.
    __device__ __forceinline__ void walk_in_turns()
    {
        const int group = tid / L, ngroups = nthr / L;
        int k = 0;
#pragma unroll 1
        for (int step = 1; step <= n; ++step) {
            const bool upd = (step % A.period) == 0;
#pragma unroll 1
            for (int base = 0; base < ml; base += ngroups) {
                const bool on = base + group < ml;
                const int al = on ? base + group : 0, a = a0 + al;
                uint32_t* vis = vis_base + (size_t)al * Wp;
                const uint32_t c = s_cur[al];
                const uint32_t u = node_id(c);
                uint32_t nx = s_start[al];
                float t_edge = tau0;
                if (step < n) {
                    load_city(u);
                    load_cand_trails(u);
                    check_row(kNoCity, vis);
                    const bool need = on && fb != 0;
                    if (G.any_group(need)) {
                        fallback(c, vis, need);
                        fallback_trails(u, need);
                    }
                    read_record(u, INT_MAX, R);
                    match(R);
                    const uint4 x = philox4x32_10(make_uint4(it, (uint32_t)a, (uint32_t)step, inst), A.key0, A.key1);
                    nx = select(c, vis, unit24(x.x), unit24(x.y), 0, on, t_edge);
                    __syncwarp();
                    if (on && gl == 0) {
                        vis[nx >> 21] |= 1u << ((nx >> 16) & 31);
                        tours[(size_t)a * n + step] = (int)node_id(nx);
                    }
                } else if constexpr (!SPM) {
                    stage_closing(u, nx);
                    t_edge = G.shfl(tv[0], 0);
                }
                __syncwarp();
                if (on && gl == 0) s_cur[al] = nx;
                if (upd && on) {
                    Entry* e = list(k + 1) + a;
                    Entry x;
                    const uint32_t key = edge_key(u, node_id(nx));
                    if constexpr (SPM) x = key;
                    else x = make_uint2(key, __float_as_uint(t_edge));
#pragma unroll 1
                    for (int r = gl; r < C; r += L) *(ALONE ? e : cg::this_cluster().map_shared_rank(e, r)) = x;
                    if (ALONE && gl == 0) hang(k + 1, a, key);
                }
                __syncwarp();
            }
            if (!upd) continue;
            sync_all();
            ++k;
            const Entry* E = list(k);
            if constexpr (!ALONE) {
#pragma unroll 1
                for (int j = tid; j < m; j += nthr) hang(k, j, key_of(E[j]));
                __syncthreads();
            }
            if constexpr (SPM) {
                update_records(k);
            } else {
#pragma unroll 1
                for (int base = 0; base < ml; base += ngroups) {
                    const bool on = base + group < ml;
                    const int al = on ? base + group : 0, a = a0 + al;
                    const uint32_t v = node_id(s_cur[al]);
                    fold_edge(k, a, other_end(key_of(E[a]), v), v, on);
                    __syncwarp();
                }
            }
            sync_all();
        }
    }

    // Evaluation, best-so-far, global update (Alg. 1). False when a wait of the
    // cluster gave up: the tours are not complete, nothing is evaluated.
    __device__ __forceinline__ bool finish(int b)
    {
        if (n_fb) atomicAdd(&misc->stat[0], (unsigned long long)n_fb);
        if (n_hit) atomicAdd(&misc->stat[1], (unsigned long long)n_hit);
        if (n_miss) atomicAdd(&misc->stat[2], (unsigned long long)n_miss);
        sync_all();   // tours and every update are visible cluster-wide
        if constexpr (!ALONE) {
            if (split && misc->stop) {
                // every CTA was told before its barrier. The edges that were
                // sent land within a few microseconds; 100 are waited for them
                // before a CTA's shared memory may go.
                const unsigned long long t0 = global_ns();
                for (int i = 0; i < (1 << 20) && global_ns() - t0 < 100000ull; ++i) {}
                sync_all();
                return false;
            }
        }

        // ---- tour lengths, a warp per ant
        const int warp = tid >> 5, warps = nthr >> 5;
#pragma unroll 1
        for (int al = warp; al < ml; al += warps) {
            const int32_t* t = tours + (size_t)(a0 + al) * n;
            long long sum = 0;
#pragma unroll 4
            for (int i = lane; i < n; i += 32) {
                const int x = __ldcg(t + i), y = __ldcg(t + (i + 1 < n ? i + 1 : 0));
                sum += euc2d(__ldg(xy + x), __ldg(xy + y));
            }
            __syncwarp();
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            if (lane == 0) {
                s_len[al] = sum;
                A.lens[A.desc[b].ant_off + a0 + al] = sum;
            }
        }
        sync_all();
        if (tid < 32) {
            long long bl = 0x7fffffffffffffffll;
            int ba = 0x7fffffff;
#pragma unroll 1
            for (int a = tid; a < m; a += 32) {
                const int r = a / mc;
                const long long l = (ALONE ? s_len : cg::this_cluster().map_shared_rank(s_len, r))[a - r * mc];
                if (l < bl || (l == bl && a < ba)) { bl = l; ba = a; }
            }
#pragma unroll 1
            for (int off = 16; off >= 1; off >>= 1) {
                const long long ol = __shfl_xor_sync(0xffffffffu, bl, off);
                const int oa = __shfl_xor_sync(0xffffffffu, ba, off);
                if (ol < bl || (ol == bl && oa < ba)) { bl = ol; ba = oa; }
            }
            if (tid == 0) {
                misc->improved = bl < misc->best_len ? 1 : 0;
                if (misc->improved) misc->best_len = bl;
                misc->bestant = ba;
            }
        }
        __syncthreads();
        if (misc->improved) {
            // the cluster copies the new best tour, one slice per CTA
            const int32_t* src = tours + (size_t)misc->bestant * n;
            for (int i = rank * nthr + tid; i < n; i += C * nthr) best[i] = __ldcg(src + i);
        }
        sync_all();

        // ---- global update on the best-so-far tour (eq. global_update)
        const float delta = __double2float_rn(1.0 / (double)misc->best_len);
        if constexpr (!SPM) {
            // a warp per edge: both halves, the candidate rows that hold the
            // edge, and the list of changed trails of a row that does not
#pragma unroll 1
            for (int i = rank * warps + warp; i < n; i += C * warps) {
                const uint32_t u = (uint32_t)__ldcg(best + i);
                const uint32_t v = (uint32_t)__ldcg(best + (i + 1 < n ? i + 1 : 0));
                const float t2 = global_rule(__ldcg(tau + at(u, v)), delta, A.rho);
                __syncwarp();
                if (lane < 2) tau[lane ? at(v, u) : at(u, v)] = t2;
#pragma unroll 1
                for (int side = 0; side < 2; ++side) {
                    const uint32_t r = side ? v : u, x = side ? u : v;
                    const bool in = lane < cl && node_id(__ldg(rows + r * 32u + lane).x) == x;
                    if (in) tauc[r * 32u + lane] = t2;
                    if (__any_sync(0xffffffffu, in)) continue;
                    if (__ldcg(tl_cnt + r) > kChanged) continue;
                    // free places hold ~0; the one node that packs to ~0 (the
                    // last of 65536) may be listed twice, which changes no result
                    const uint32_t px = pack(x);
                    const bool has = px != 0xffffffffu && __ldcg(tl + r * 32u + lane) == px;
                    if (!(t2 >= tau0)) {
                        // below tau0 (only from a restored state): the row's
                        // full scan must read every trail
                        if (lane == 0) atomicMax(tl_cnt + r, kReadAll);
                    } else if (!__any_sync(0xffffffffu, has) && lane == 0 &&
                               __float_as_uint(t2) != __float_as_uint(tau0)) {
                        const int to = atomicAdd(tl_cnt + r, 1);
                        if (to < kChanged) tl[r * 32u + to] = px;
                    }
                }
            }
        } else {
            // record best[i] sees, in tour order, the edge (best[i-1], best[i])
            // then (best[i], best[i+1]); record best[0] sees edge 0 then edge
            // n-1. Every record is on the tour: its latest working copy goes
            // back to the context's arrays with the two updates applied.
            unsigned long long h = 0, miss = 0;
#pragma unroll 1
            for (int i = rank * nthr + tid; i < n; i += C * nthr) {
                const int r = __ldcg(best + i);
                const int prev = __ldcg(best + (i > 0 ? i - 1 : n - 1));
                const int nxt = __ldcg(best + (i + 1 < n ? i + 1 : 0));
                const uint2* Q = rec_of((uint32_t)r);
                uint2 meta = ld_rec(Q + s_slots * NC);
                int cp = 0;
                for (int x = 1; x < NC; ++x) {
                    const uint2 y = ld_rec(Q + s_slots * NC + x);
                    if ((int)y.y > (int)meta.y) {
                        meta = y;
                        cp = x;
                    }
                }
                int32_t* oi = sidx + (size_t)r * s_slots;
                float* ov = tau + (size_t)r * s_slots;
                int tail = (int)meta.x;
#pragma unroll 4
                for (int q = 0; q < s_slots; ++q) {
                    const uint2 x = ld_rec(Q + q * NC + cp);
                    oi[q] = (int32_t)x.x;
                    ov[q] = __uint_as_float(x.y);
                }
                // Alg. 3 twice
#pragma unroll 1
                for (int e = 0; e < 2; ++e) {
                    const int nb = (e == 0) == (i > 0) ? prev : nxt;
                    int hit = -1;
#pragma unroll 4
                    for (int q = 0; q < s_slots; ++q)
                        if (oi[q] == nb) hit = q;
                    if (hit >= 0) {
                        ov[hit] = global_rule(ov[hit], delta, A.rho);
                        ++h;
                    } else {
                        tail = tail + 1 == s_slots ? 0 : tail + 1;
                        oi[tail] = nb;
                        ov[tail] = global_rule(tau0, delta, A.rho);
                        ++miss;
                    }
                }
                stail[r] = tail;
            }
            if (h) atomicAdd(&misc->stat[1], h);
            if (miss) atomicAdd(&misc->stat[2], miss);
        }
        __syncthreads();
        if (tid == 0) {
            unsigned long long* st = A.stats + 4 * (size_t)b;
            atomicAdd(st + 0, misc->stat[0]);
            if (rank == 0) atomicAdd(st + 1, (unsigned long long)m * (unsigned long long)(n - 1));
            atomicAdd(st + 2, misc->stat[1]);
            atomicAdd(st + 3, misc->stat[2]);
            if (rank == 0) {
                A.best_len[b] = misc->best_len;
                A.iteration[b] = misc->iteration + 1;
            }
        }
        sync_all();
        return true;
    }

    // The next instance of this cluster. The first ncl instances (longest
    // first) go to clusters 0..ncl-1; with a counter, a cluster that finishes
    // then takes the next untaken instance. Rank 0 draws it; each CTA's thread
    // 0 copies it from rank 0's shared memory between two cluster barriers (the
    // second keeps rank 0 from rewriting it or exiting before every CTA has
    // read it), and the CTA reads its own copy.
    __device__ __forceinline__ int next_instance(int oi, int ncl)
    {
        if (!A.sched) return oi + ncl;
        // (after a wait of any cluster gave up the iteration is lost anyway)
        if (rank == 0 && tid == 0) {
            const int drawn = ncl + atomicAdd(A.sched, 1);
            misc->next = __ldcg(A.status) == kWaitGaveUp ? INT_MAX : drawn;
        }
        sync_all();
        if (tid == 0) misc->next_local = (ALONE ? misc : cg::this_cluster().map_shared_rank(misc, 0))->next;
        sync_all();
        return misc->next_local;
    }
};

}  // namespace

// MODE 0: pheromone matrix. MODE 1: SPM, the records' working copies in
// global memory. MODE 2: SPM, record r's working copies in the shared memory
// of CTA r mod C (other CTAs reach them through distributed shared memory).
// ALONE: the launch's clusters are single CTAs. One ant per group of L lanes;
// on clusters the CTA's last warp publishes.
template <int L, int MODE, bool ALONE, int KIND>
__global__ void __launch_bounds__(ALONE ? kAloneThreads : kClusterThreads, 1)
construct_kernel(const __grid_constant__ ConstructArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Colony<L, MODE, ALONE, KIND> w(A, true);
    w.open(smem);
    const int ncl = gridDim.x / w.C;
#pragma unroll 1
    for (int oi = blockIdx.x / w.C; oi < A.num_inst;) {
        const int b = A.order[oi];
        w.begin(b);
        if ((w.tid >> 5) < w.ants_warps) {
            w.walk();
        } else if constexpr (!ALONE) {
            if ((w.tid >> 5) == (w.nthr >> 5) - 1) w.publish();
        }
        w.kbase += w.n / A.period;
        if (!w.finish(b)) break;
        oi = w.next_instance(oi, ncl);
    }
}

// The same iteration with barriers between the ants' selections and the updates:
// the groups take several ants in turn when there are more, and a step's edges are
// looked up through an index.
template <int L, int MODE, bool ALONE>
__global__ void __launch_bounds__(ALONE ? kAloneThreads : kClusterAntThreads, 1)
construct_turns_kernel(const __grid_constant__ ConstructArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Colony<L, MODE, ALONE, kTurns> w(A, false);
    w.open(smem);
    const int ncl = gridDim.x / w.C;
#pragma unroll 1
    for (int oi = blockIdx.x / w.C; oi < A.num_inst;) {
        const int b = A.order[oi];
        w.begin(b);
        w.walk_in_turns();
        w.finish(b);
        oi = w.next_instance(oi, ncl);
    }
}

// the kernel of this variant for a number of lanes per ant
template <int MODE, bool ALONE, int KIND>
void* construct_variant(int lanes)
{
    if constexpr (KIND == kTurns) {
        switch (lanes) {
        case 8: return reinterpret_cast<void*>(construct_turns_kernel<8, MODE, ALONE>);
        case 16: return reinterpret_cast<void*>(construct_turns_kernel<16, MODE, ALONE>);
        default: return nullptr;
        }
    } else {
        switch (lanes) {
        case 4: return reinterpret_cast<void*>(construct_kernel<4, MODE, ALONE, KIND>);
        case 8: return reinterpret_cast<void*>(construct_kernel<8, MODE, ALONE, KIND>);
        case 16: return reinterpret_cast<void*>(construct_kernel<16, MODE, ALONE, KIND>);
        case 32: return reinterpret_cast<void*>(construct_kernel<32, MODE, ALONE, KIND>);
        default: return nullptr;
        }
    }
}

}  // namespace acs
