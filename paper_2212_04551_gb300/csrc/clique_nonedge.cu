// clique_nonedge.cu -- k-clique counting over a whole graph by branching on
// non-edges (clique_nonedge.cuh): the count of Algorithm 4 (clique counting)
// without visiting the cliques one by one.
//
// Every clique is counted at its root, its lowest vertex in the (degree, id)
// orientation, inside the root's out-neighbourhood N+(r).  Two launches share
// the roots by d = |N+(r)|:
//
//   * k_clique_ne_light, d <= 32: one warp per root.  The bit rows are one
//     word each, one per lane, and the whole of N+(r) is one candidate set.
//   * k_clique_ne_heavy, 32 < d <= 1,024: one block per root.  Its warps build
//     the symmetric bit rows of N+(r) together in shared memory (positions in
//     orientation order) and then take the root's children p -- candidates:
//     the neighbours of p after p -- one by one from a counter of the root in
//     global memory.  The root list is gone through again for the largest
//     roots, so that blocks without a root of their own join one that is
//     still at work (they build its rows again and draw on the same counter).
//     A child's members without non-edges are set aside as a number; the
//     others are re-indexed (up to 128 of them) and counted in registers.
//     From a set with more, members are first taken out one by one in shared
//     memory, by the same rule, until 128 are left (ne_wide_step), unless three
//     sizes are to go and nearly all would have to be (ne_wide_direct).
//
// The row build reads every out-list of N+(r) once: eight lanes per list with
// 16-byte loads (the lists are padded and aligned for it), each entry tested
// against a small hash filter of N+(r) before it is searched in the list.
//
// Roots above 1,024 are the list path's (clique_list.cu).
//
// What bounds it: the heavy launch, instruction issue and instruction fetch
// (issue slots 0.49 busy, `no_instruction` the first stall; 2.1e10 warp
// instructions at k = 4..7 on the Chung-Lu graph of 10^6 vertices, where the
// walk over the cliques took 9.5e11).  Loops whose trip count depends on data
// are therefore not unrolled: with the compiler's unrolling an earlier state of
// the heavy kernel was 401 KB of code instead of 113 KB, and 81 ms instead of 46.  The light
// launch is bound by the latency of its chain of dependent loads per root.
// Measured, whole call on that graph: k = 4..7 1,378 -> 35 ms, k = 4 8.0 ->
// 2.8 ms; block-model graph of 2,000 vertices, k = 6..12: 20.9 -> 0.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "clique_nonedge.cuh"
#include "common.cuh"

namespace gpm {

constexpr int NE_LIGHT_D = 32;
constexpr int NE_LIGHT_WARPS = 8;     // warps per block of the light launch
constexpr int NE_LIGHT_GRAB = 8;      // roots a warp takes at a time
constexpr int NE_WARPS = 4;           // warps per block of the heavy launch
constexpr int NE_HELP_D = 128;        // roots above this are offered to further blocks ...
constexpr int NE_HELP_ROUNDS = 24;    // ... this many times (k >= 6, where a child's work can be large)
constexpr int NE_SCRATCH = 64 + 128;   // words for a second re-indexing (ne_four_again)
constexpr int NE_DIRECT_M = 160;      // wide sets of three sizes to go: from this many members with non-edges,
constexpr int NE_DIRECT_E = 2;        // and this many on average, the triangles are counted (ne_wide_direct)
constexpr int NE_FILTER_WORDS = 64;   // hash filter of N+(r): 2,048 bits

struct NeLaunch {
    const int32_t* __restrict__ off;
    const int32_t* __restrict__ adj;
    const int32_t* __restrict__ outdeg;
    const int32_t* __restrict__ deg;
    const int32_t* __restrict__ roots;    // heaviest out-degree first
    long long first, last;                // this launch's positions in roots
    long long n_help;                     // of these, the first n_help are offered again ...
    int rounds;                           // ... rounds times
    int grab;                             // children a warp takes at a time
    int maxd, w, ws;                      // heavy: largest d, its words, the row stride (odd)
    int warp_words;                       // heavy: shared words per warp
    unsigned int* next_child;             // heavy: per position, the next child not yet taken
    unsigned int* tri;                    // nullable: triangles per out-list entry (rounds = 0)
    NeParams ne;
    Control* ctl;
    unsigned long long* busy;             // this launch's warp time
    unsigned long long* ticket;           // next position (light) or root offer (heavy)
};

__device__ __forceinline__ unsigned ne_hash(int x) { return (unsigned)x * 2654435761u; }

// End of a block: its warps' counts are added up in shared memory first (one
// global add per size and block; thousands of warps would queue on each).
__device__ __forceinline__ void ne_finish(const NeLaunch& p, NeCount& c, unsigned long long units,
                                          unsigned long long busy, int lane) {
    const NeParams& ne = p.ne;
    Control* ctl = p.ctl;
    __shared__ unsigned long long sum[NE_LEVELS + 3];
    ne_fold(ne, c, lane);
    if (threadIdx.x < NE_LEVELS + 3) sum[threadIdx.x] = 0ull;
    __syncthreads();
    if (c.ovf) atomicExch(&ctl->overflow, 1);
    if (lane >= ne.k_lo && lane <= ne.k_hi) gpm_atomic_add_cc(&sum[lane], c.size, &ctl->overflow);
    if (lane == 0) {
        atomicAdd(&sum[NE_LEVELS], units);
        atomicAdd(&sum[NE_LEVELS + 1], c.wops);
        atomicAdd(&sum[NE_LEVELS + 2], busy);
    }
    __syncthreads();
    const int t = threadIdx.x;
    if (t < NE_LEVELS) gpm_atomic_add_cc(&ctl->counts[t], sum[t], &ctl->overflow);
    else if (t < NE_LEVELS + 3 && sum[t])
        atomicAdd(t == NE_LEVELS ? &ctl->units_done : t == NE_LEVELS + 1 ? &ctl->word_ops : p.busy, sum[t]);
}

// ------------------------------------------------------------------- light

__global__ void __launch_bounds__(NE_LIGHT_WARPS * 32) k_clique_ne_light(NeLaunch p) {
    struct Warp {
        int32_t list[32];
        uint32_t g[32];
        uint32_t h[32];
        uint32_t filter[32];
        uint32_t stk[NE_LEVELS];
    };
    __shared__ Warp sh[NE_LIGHT_WARPS];
    Warp& W = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int sub = lane & 7, grp = lane >> 3;
    NeCount c;
    unsigned long long units = 0, busy = 0;
    const unsigned long long t0 = gpm_globaltimer();
#pragma unroll 1
    for (;;) {
        unsigned long long pos = 0;
        if (lane == 0) pos = p.first + atomicAdd(p.ticket, (unsigned long long)NE_LIGHT_GRAB);
        pos = __shfl_sync(GPM_FULL_MASK, pos, 0);
        if (pos >= (unsigned long long)p.last) break;
        const int nr = (int)min((unsigned long long)NE_LIGHT_GRAB, (unsigned long long)p.last - pos);
        // the batch's roots, one per lane
        int my_d = 0, my_off = 0;
        if (lane < nr) {
            const int r = p.roots[pos + lane];
            my_d = p.outdeg[r];
            my_off = p.off[r];
        }
#pragma unroll 1
        for (int q = 0; q < nr; q++) {
            const int d = __shfl_sync(GPM_FULL_MASK, my_d, q);
            const int beg = __shfl_sync(GPM_FULL_MASK, my_off, q);
            int ub = 0, du = 0;
            W.g[lane] = 0u;
            W.filter[lane] = 0u;
            __syncwarp();
            if (lane < d) {
                const int u = p.adj[beg + lane];
                W.list[lane] = u;
                const unsigned hu = ne_hash(u) >> 22;
                atomicOr(&W.filter[hu >> 5], 1u << (hu & 31));
                ub = p.off[u];
                du = p.outdeg[u];
            } else {
                W.list[lane] = INT32_MAX;
            }
            __syncwarp();
#pragma unroll 1
            for (int i0 = 0; i0 < d; i0 += 4) {
                const int i = min(i0 + grp, 31);
                const int b = __shfl_sync(GPM_FULL_MASK, ub, i);
                const int len = __shfl_sync(GPM_FULL_MASK, du, i);   // 0 from d on
#pragma unroll 1
                for (int t = 4 * sub; t < len; t += 32) {
                    const int4 v = *reinterpret_cast<const int4*>(p.adj + b + t);   // 16-byte aligned, padded
                    const int xs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int z = 0; z < 4; z++) {
                        const int x = xs[z];
                        const unsigned hx = ne_hash(x) >> 22;
                        if (!((W.filter[hx >> 5] >> (hx & 31)) & 1u)) continue;
                        int lo = 0;
#pragma unroll
                        for (int step = 16; step > 0; step >>= 1) lo += W.list[lo + step - 1] < x ? step : 0;
                        if (lo < d && W.list[lo] == x) {
                            atomicOr(&W.g[i], 1u << lo);
                            atomicOr(&W.g[lo], 1u << i);
                            if (p.tri) {
                                atomicAdd(&p.tri[beg + i], 1u);
                                atomicAdd(&p.tri[beg + lo], 1u);
                                atomicAdd(&p.tri[b + t + z], 1u);
                            }
                        }
                    }
                }
            }
            __syncwarp();
            const uint32_t all = d >= 32 ? 0xffffffffu : (1u << d) - 1u;
            const uint32_t row = W.g[lane];
            const int rem = p.ne.k_hi - 1;
            if (rem == 2) {
                const unsigned e2 = __reduce_add_sync(GPM_FULL_MASK, lane < d ? (unsigned)(d - 1 - __popc(row)) : 0u);
                ne_pairs(p.ne, c, (unsigned)d, e2, lane);
            } else {
                W.h[lane] = all & ~row & ~(1u << lane);
                __syncwarp();
                ne_sets<1>(p.ne, c, d, 0, 1, W.h, W.stk, nullptr, lane);
                __syncwarp();
            }
        }
        units += (unsigned)nr;
    }
    busy = gpm_globaltimer() - t0;
    ne_finish(p, c, units, busy, lane);
}

// ------------------------------------------------------------------- heavy

// shared words of one warp: a candidate bitmap per level, the member lists
// (16-bit positions; of the current set, and of a wide set with the non-edges
// of each), the re-indexed rows and their level stack
__host__ __device__ inline int ne_warp_words(int maxd, int w, bool deep) {
    if (!deep) return 3 * w + ((maxd + 3) & ~3) / 2;
    return NE_LEVELS * w + 3 * ((maxd + 3) & ~3) / 2 + 32 * NE_W * NE_W + NE_W * NE_LEVELS + NE_SCRATCH;
}

__host__ __device__ inline int ne_block_words(int maxd, int ws) {
    return 2 * ((maxd + 3) & ~3) + NE_FILTER_WORDS + maxd * ws + 4;
}

struct NeWarp {
    uint32_t* cand;     // [level][w]
    uint16_t* mem;      // members of the current set; then those with a non-edge
    uint16_t* wide;     // members of the wide set being taken apart ...
    uint16_t* we;       // ... and their non-edges in it (NE_GONE: taken out)
    uint32_t* Hs;
    uint32_t* stk;
    uint32_t* scratch;
};
constexpr unsigned NE_GONE = 0xffffu;

// rows of H among the m members mem[], ceil(m/32) of W words used
template <int W>
__device__ __forceinline__ void ne_reindex(const uint32_t* rows, int ws, const uint16_t* mem, int m, uint32_t* Hs, int lane) {
    int pm[W];
#pragma unroll
    for (int b = 0; b < W; b++) pm[b] = 32 * b + lane < m ? mem[32 * b + lane] : -1;
#pragma unroll 1
    for (int i = 0; i < m; i++) {
        const int pi = mem[i];
        const uint32_t* row = rows + pi * ws;
#pragma unroll
        for (int b = 0; b < W; b++) {
            const bool non = pm[b] >= 0 && pm[b] != pi && !((row[pm[b] >> 5] >> (pm[b] & 31)) & 1u);
            const uint32_t word = __ballot_sync(GPM_FULL_MASK, non);
            if (lane == b) Hs[i * W + b] = word;
        }
    }
    __syncwarp();
}

// the m <= 128 members mem[] with non-edges, `a` members without, three sizes
// or more to go
__device__ __forceinline__ void ne_indexed(const NeLaunch& p, NeCount& c, const NeWarp& k, const uint32_t* rows, int m,
                                           int a, int h, int lane) {
    if (m <= 32) {
        ne_reindex<1>(rows, p.ws, k.mem, m, k.Hs, lane);
        ne_sets<1>(p.ne, c, m, a, h, k.Hs, k.stk, k.scratch, lane);
    } else {
        ne_reindex<NE_W>(rows, p.ws, k.mem, m, k.Hs, lane);
        ne_sets<NE_W>(p.ne, c, m, a, h, k.Hs, k.stk, k.scratch, lane);
    }
    __syncwarp();
}

// the set bits of C (w words) into list[], ascending; returns how many
__device__ __forceinline__ int ne_members(const uint32_t* C, int w, uint16_t* list, int lane) {
    int n = 0;
#pragma unroll 1
    for (int q = 0; q < w; q++) {
        const uint32_t word = C[q];
        if ((word >> lane) & 1u) list[n + __popc(word & gpm_lanemask_lt())] = (uint16_t)(32 * q + lane);
        n += __popc(word);
    }
    __syncwarp();
    return n;
}

// non-edges of position pos within C (which holds it)
__device__ __forceinline__ int ne_degree(const uint32_t* rows, int ws, int w, const uint32_t* C, int pos) {
    const uint32_t* row = rows + pos * ws;
    int e = -1;                                       // itself
#pragma unroll 1
    for (int z = 0; z < w; z++) e += __popc(C[z] & ~row[z]);
    return e;
}

// What is left to do with a set
enum NeTodo { NE_DONE, NE_INDEX, NE_WIDE };

// The set C (w words) of a traversal of size h: counted, or (three sizes or
// more to go) its m members with non-edges in k.mem and `a` without: NE_INDEX
// up to 128 members, else NE_WIDE.
__device__ __forceinline__ NeTodo ne_node(const NeLaunch& p, NeCount& c, const NeWarp& k, const uint32_t* rows, int w,
                                          const uint32_t* C, int h, int& m, int& a, int lane) {
    const int n = ne_members(C, w, k.mem, lane);
    if (h + n < p.ne.k_lo) return NE_DONE;
    const int rem = p.ne.k_hi - h;
    if (rem == 1) {
        c.size = gpm_add_cc(c.size, lane == p.ne.k_hi ? (unsigned)n : lane == h ? 1u : 0u, c.ovf);
        return NE_DONE;
    }
    // non-edges of every member; those that have one move to the front
    unsigned e2 = 0;
    m = 0;
#pragma unroll 1
    for (int t0 = 0; t0 < n; t0 += 32) {
        const int t = t0 + lane;
        int e = 0, pos = 0;
        if (t < n) {
            pos = k.mem[t];
            e = ne_degree(rows, p.ws, w, C, pos);
        }
        e2 += (unsigned)e;
        const unsigned bal = __ballot_sync(GPM_FULL_MASK, e > 0);   // every lane has read its entry
        if (e > 0) k.mem[m + __popc(bal & gpm_lanemask_lt())] = (uint16_t)pos;
        m += __popc(bal);
        __syncwarp();
    }
    c.wops += (unsigned)(n * w);
    if (rem == 2) {
        ne_pairs(p.ne, c, (unsigned)n, __reduce_add_sync(GPM_FULL_MASK, e2), lane);
        return NE_DONE;
    }
    a = n - m;
    if (m == 0) {
        ne_matching(p.ne, c, h, n, 0, lane);
        return NE_DONE;
    }
    return m <= 32 * NE_W ? NE_INDEX : NE_WIDE;
}

// Three sizes to go, a wide set C with m members that have non-edges: where
// these leave little to a closed form -- taken out one by one, nearly all would
// have to go -- the triangles of the graph among C are counted directly, as the
// walk counts them.  Returns their number, the edges and the members (28, 20
// and 12 bits from the lowest), 0 if the set is better taken apart.  CU: w words
// of scratch.  Out of line: the code of the other sets is bound by its fetch.
//
// 5-cliques, walk / taken apart / this where it applies: complete multipartite graphs,
// 600 vertices in parts of 100 47 / 91 / 33 ms, in parts of 5 103 / 217 / 80, in
// parts of 2 66 / 2.4 / 2.7; G(600, 0.8) 41 / 67 / 26, G(900, 0.7) 93 / 126 / 43.
// From 129, 160 or 200 members: parts of 50, 300 vertices, k = 5 3.8 / 3.7 / 5.0,
// k = 6 11.0 / 8.8 / 8.8.
__device__ __noinline__ unsigned long long ne_wide_direct(const uint32_t* rows, int ws, int w, const uint32_t* C,
                                                          uint32_t* CU, uint16_t* mem, int m, int lane) {
    const int n = ne_members(C, w, mem, lane);
    unsigned e2 = 0;
    for (int t = lane; t < n; t += 32) e2 += (unsigned)ne_degree(rows, ws, w, C, mem[t]);
    e2 = __reduce_add_sync(GPM_FULL_MASK, e2);
    if (e2 < (unsigned)(NE_DIRECT_E * m)) return 0;
    unsigned t = 0;
    for (int i = 0; i < n - 2; i++) {
        const int u = mem[i];
        const uint32_t* ru = rows + u * ws;
        if (lane < w) CU[lane] = C[lane] & ru[lane];
        __syncwarp();
        for (int j = i + 1 + lane; j < n; j += 32) {
            const int v = mem[j];
            if (!((CU[v >> 5] >> (v & 31)) & 1u)) continue;
            const uint32_t* rv = rows + v * ws;
            t += __popc(CU[v >> 5] & rv[v >> 5] & (0xfffffffeu << (v & 31)));
#pragma unroll 4
            for (int z = (v >> 5) + 1; z < w; z++) t += __popc(CU[z] & rv[z]);
        }
        __syncwarp();
    }
    t = __reduce_add_sync(GPM_FULL_MASK, t);
    return (unsigned long long)t | (unsigned long long)((unsigned)n * (n - 1) - e2) / 2 << 28 | (unsigned long long)n << 48;
}

// One step on the wide set C of traversal size lv (its members in k.wide,
// `left` of n not taken out yet): NE_DONE if it is finished, NE_INDEX if at
// most 128 members with non-edges are left (now in k.mem), else NE_WIDE: the
// member with the most non-edges is taken out of C, and N is the set that
// holds it.
__device__ __forceinline__ NeTodo ne_wide_step(const NeLaunch& p, NeCount& c, const NeWarp& k, const uint32_t* rows,
                                               int w, uint32_t* C, uint32_t* N, int lv, int n, int& left, int& m,
                                               int& a, int lane) {
    unsigned key = 0, sum = 0;
    m = 0;
#pragma unroll 1
    for (int t0 = 0; t0 < n; t0 += 32) {
        const unsigned e = t0 + lane < n ? k.we[t0 + lane] : NE_GONE;
        const bool some = e != NE_GONE && e > 0;
        const unsigned bal = __ballot_sync(GPM_FULL_MASK, some);
        if (some) {
            key = max(key, (e << 10) | (unsigned)(t0 + lane));
            sum += e;
            k.mem[m + __popc(bal & gpm_lanemask_lt())] = k.wide[t0 + lane];
        }
        m += __popc(bal);
    }
    __syncwarp();
    if (lv + left < p.ne.k_lo) return NE_DONE;
    a = left - m;
    key = __reduce_max_sync(GPM_FULL_MASK, key);
    if ((key >> 10) <= 1) {
        ne_matching(p.ne, c, lv, left, (int)__reduce_add_sync(GPM_FULL_MASK, sum) / 2, lane);
        return NE_DONE;
    }
    if (m <= 32 * NE_W) return NE_INDEX;
    const int i = (int)(key & 1023u);
    const int v = k.wide[i];
    const uint32_t* row = rows + v * p.ws;
    if (lane < w) {
        const uint32_t x = lane == (v >> 5) ? C[lane] & ~(1u << (v & 31)) : C[lane];
        C[lane] = x;
        N[lane] = x & row[lane];
    }
#pragma unroll 1
    for (int t = lane; t < n; t += 32) {
        const unsigned e = k.we[t];
        const int u = k.wide[t];
        if (t == i) k.we[t] = (uint16_t)NE_GONE;
        else if (e != NE_GONE && !((row[u >> 5] >> (u & 31)) & 1u)) k.we[t] = (uint16_t)(e - 1);
    }
    left--;
    __syncwarp();
    return NE_WIDE;
}

// All cliques of the set in cand[2] (traversals of size 2), depth first over
// wide sets.  DIRECT: with the call of ne_wide_direct, around which the loops
// keep fewer values in registers (Chung-Lu, 10^6 vertices, k = 5 without / with:
// 5.91 / 6.07 ms, k = 4..7 33.9 / 33.4).
template <bool DIRECT>
__device__ __forceinline__ void ne_child(const NeLaunch& p, NeCount& c, const NeWarp& k, const uint32_t* rows, int w,
                                         int lane) {
    int h = 2;                 // the size of the set looked at
    int lv = 1;                // the innermost wide set (1: none; those above it are wide too)
    int n = 0, left = 0, m = 0, a = 0;
#pragma unroll 1
    for (;;) {
        NeTodo todo = ne_node(p, c, k, rows, w, k.cand + h * w, h, m, a, lane);
        if (DIRECT && todo == NE_WIDE && h + 3 == p.ne.k_hi && m >= NE_DIRECT_M) {
            const unsigned long long r = ne_wide_direct(rows, p.ws, w, k.cand + h * w, k.cand + (h + 1) * w, k.mem, m, lane);
            if (r) {
                const int j = lane - h;                // cliques of h + j members
                c.size = gpm_add_cc(c.size, j == 3 ? r & 0xfffffffu : j == 2 ? (r >> 28) & 0xfffffu : j == 1 ? r >> 48
                                            : j == 0 ? 1ull : 0ull, c.ovf);
                todo = NE_DONE;
            }
        }
        bool load = todo == NE_WIDE, over = false;
        if (load) lv = h;
#pragma unroll 1
        for (;;) {
            if (todo == NE_INDEX) {
                ne_indexed(p, c, k, rows, m, a, h, lane);
                if (lv >= 2) ne_settle(p.ne, c, lane);
            }
            if (over) {        // nothing is left of the wide set
                lv--;
                load = true;
            }
            if (lv < 2) return;
            uint32_t* C = k.cand + lv * w;
            if (load) {        // its members and their non-edges
                n = left = ne_members(C, w, k.wide, lane);
#pragma unroll 1
                for (int t = lane; t < n; t += 32) k.we[t] = (uint16_t)ne_degree(rows, p.ws, w, C, k.wide[t]);
                __syncwarp();
                c.wops += (unsigned)(n * w);
                load = false;
            }
            todo = ne_wide_step(p, c, k, rows, w, C, C + w, lv, n, left, m, a, lane);
            over = todo != NE_WIDE;
            h = over ? lv : lv + 1;
            if (!over) break;
        }
    }
}

// DEEP: three sizes or more to go below a child (k >= 5); without, neither the
// re-indexed rows nor their registers are there (48 instead of 96), and twice
// the warps are resident: k = 4 on the Chung-Lu graph 4.0 -> 2.8 ms.
template <bool DEEP, bool DIRECT>
__global__ void __launch_bounds__(NE_WARPS * 32, DEEP ? 5 : 10) k_clique_ne_heavy(NeLaunch p) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ unsigned long long s_pos;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int dpad = (p.maxd + 3) & ~3;
    int* list = reinterpret_cast<int*>(smem);
    int* pos = list + dpad;
    uint32_t* filter = reinterpret_cast<uint32_t*>(pos + dpad);
    uint32_t* rows = filter + NE_FILTER_WORDS;
    uint32_t* mine = smem + ne_block_words(p.maxd, p.ws) + wib * p.warp_words;
    NeWarp k;
    k.cand = mine;
    if (DEEP) {
        k.Hs = k.cand + NE_LEVELS * p.w;
        k.stk = k.Hs + 32 * NE_W * NE_W;
        k.scratch = k.stk + NE_W * NE_LEVELS;
        k.mem = reinterpret_cast<uint16_t*>(k.scratch + NE_SCRATCH);
        k.wide = k.mem + dpad;
        k.we = k.wide + dpad;
    } else {
        k.Hs = k.stk = k.scratch = nullptr;
        k.mem = reinterpret_cast<uint16_t*>(k.cand + 3 * p.w);
        k.wide = k.we = nullptr;
    }
    const unsigned long long n_own = (unsigned long long)(p.last - p.first);
    const unsigned long long n_offers = n_own + (unsigned long long)p.n_help * p.rounds;
    NeCount c;
    unsigned long long units = 0, busy = 0;
#pragma unroll 1
    for (;;) {
        __syncthreads();                  // the rows of the last root are no longer read
        if (threadIdx.x == 0) {
            // the next offer whose root has children left
            unsigned long long found = ~0ull;
#pragma unroll 1
            for (;;) {
                const unsigned long long t = atomicAdd(p.ticket, 1ull);
                if (t >= n_offers) break;
                const unsigned long long i = t < n_own ? t : (t - n_own) % (unsigned long long)p.n_help;
                if (t < n_own || *(volatile unsigned int*)&p.next_child[i] < (unsigned)p.outdeg[p.roots[p.first + i]]) {
                    found = i;
                    break;
                }
            }
            s_pos = found;
        }
        __syncthreads();
        const unsigned long long at = s_pos;
        if (at == ~0ull) break;
        const unsigned long long t_unit = gpm_globaltimer();
        const int r = p.roots[p.first + at];
        const int d = p.outdeg[r], beg = p.off[r];
        const int w = (d + 31) >> 5;
        // ---- the rows: ids and sort keys, ranks, then the out-lists of N+(r)
#pragma unroll 1
        for (int t = threadIdx.x; t < d; t += blockDim.x) {
            const int u = p.adj[beg + t];
            list[t] = u;
            rows[t] = (uint32_t)p.deg[u];
        }
#pragma unroll 1
        for (int t = threadIdx.x; t < NE_FILTER_WORDS; t += blockDim.x) filter[t] = 0u;
        __syncthreads();
#pragma unroll 1
        for (int t = threadIdx.x; t < d; t += blockDim.x) {
            const uint32_t kt = rows[t];
            int rank = 0;
#pragma unroll 1
            for (int s = 0; s < d; s++) {
                const uint32_t ks = rows[s];
                rank += (ks < kt || (ks == kt && s < t)) ? 1 : 0;
            }
            pos[t] = rank;
            const unsigned hu = ne_hash(list[t]) >> 21;
            atomicOr(&filter[hu >> 5], 1u << (hu & 31));
        }
        __syncthreads();
#pragma unroll 1
        for (int t = threadIdx.x; t < d * p.ws; t += blockDim.x) rows[t] = 0u;
        __syncthreads();
#pragma unroll 1
        for (int i = threadIdx.x >> 3; i < d; i += NE_WARPS * 4) {
            const int u = list[i];
            const int b = p.off[u], len = p.outdeg[u];
            const int pi = pos[i];
#pragma unroll 1
            for (int t = 4 * (lane & 7); t < len; t += 32) {
                const int4 v = *reinterpret_cast<const int4*>(p.adj + b + t);   // 16-byte aligned, padded
                const int xs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int z = 0; z < 4; z++) {
                    const int x = xs[z];
                    const unsigned hx = ne_hash(x) >> 21;
                    if (!((filter[hx >> 5] >> (hx & 31)) & 1u)) continue;
                    int lo = 0, hi = d - 1;
#pragma unroll 1
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (list[mid] < x) lo = mid + 1; else hi = mid;
                    }
                    if (list[lo] == x) {
                        const int px = pos[lo];
                        atomicOr(&rows[pi * p.ws + (px >> 5)], 1u << (px & 31));
                        atomicOr(&rows[px * p.ws + (pi >> 5)], 1u << (pi & 31));
                        if (p.tri) {
                            atomicAdd(&p.tri[beg + i], 1u);
                            atomicAdd(&p.tri[beg + lo], 1u);
                            atomicAdd(&p.tri[b + t + z], 1u);
                        }
                    }
                }
            }
        }
        __syncthreads();
        // ---- the children: traversals (r, q) of size 2
#pragma unroll 1
        for (;;) {
            unsigned first = 0;
            if (lane == 0) first = atomicAdd(&p.next_child[at], (unsigned)p.grab);
            first = __shfl_sync(GPM_FULL_MASK, first, 0);
            if (first >= (unsigned)d) break;
            const int upto = min((int)first + p.grab, d);
#pragma unroll 1
            for (int q = (int)first; q < upto; q++) {
                // the neighbours of q after it
                uint32_t* C = k.cand + 2 * w;
                if (lane < w) {
                    const uint32_t after = lane < (q >> 5) ? 0u : lane > (q >> 5) ? 0xffffffffu
                                           : (q & 31) == 31 ? 0u : 0xffffffffu << ((q & 31) + 1);
                    C[lane] = rows[q * p.ws + lane] & after;
                }
                __syncwarp();
                if (DEEP) {
                    ne_child<DIRECT>(p, c, k, rows, w, lane);
                } else {
                    int m, a;
                    ne_node(p, c, k, rows, w, C, 2, m, a, lane);   // two sizes to go at most: counted
                }
                __syncwarp();
            }
        }
        if (DEEP) ne_fold(p.ne, c, lane);
        if (threadIdx.x == 0) units++;
        busy += gpm_globaltimer() - t_unit;
    }
    ne_finish(p, c, units, busy, lane);
}

// ------------------------------------------------------------------- host

// C(n, k), saturated, on the current device (uploaded once per device)
static const unsigned long long* device_binomials(cudaStream_t s) {
    static std::mutex mu;
    static std::map<int, unsigned long long*> tables;
    int dev = 0;
    GPM_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    auto it = tables.find(dev);
    if (it != tables.end()) return it->second;
    std::vector<unsigned long long> t((size_t)(NE_BINOM_N + 1) * NE_BINOM_K, 0ull);
    for (int n = 0; n <= NE_BINOM_N; n++)
        for (int k = 0; k < NE_BINOM_K; k++) {
            unsigned long long& x = t[(size_t)n * NE_BINOM_K + k];
            if (k == 0) x = 1;
            else if (n > 0) {
                const unsigned long long a = t[(size_t)(n - 1) * NE_BINOM_K + k - 1], b = t[(size_t)(n - 1) * NE_BINOM_K + k];
                x = a + b < a || a == ~0ull || b == ~0ull ? ~0ull : a + b;
            }
        }
    auto* d = static_cast<unsigned long long*>(upload_table(t.data(), t.size() * sizeof(t[0]), s, "binomial table"));
    tables[dev] = d;
    return d;
}

// Whole-graph clique counts of sizes k_lo .. k_hi (k_hi >= 3) into ctl (its
// counters zero); roots above the bitmap limit are left out.
void launch_clique_nonedge(gpm_graph* g, int k_lo, int k_hi, Control* ctl, Launches& made, unsigned int* tri) {
    cudaStream_t s = g->stream;
    NeLaunch p{};
    p.roots = ensure_root_order(g, GPM_APP_CLIQUE);
    p.off = g->dag_off.as<int32_t>();
    p.adj = g->dag_adj.as<int32_t>();
    p.outdeg = g->dag_outdeg.as<int32_t>();
    p.deg = g->degree.as<int32_t>();
    p.ne.k_lo = std::max(k_lo, 3);
    p.ne.k_hi = k_hi;
    p.ne.binom = device_binomials(s);
    p.ctl = ctl;
    p.tri = tri;
    // positions by out-degree: [0, above) list path, [above, big) heavy, [big, all) light
    const int need = std::max(p.ne.k_lo - 1, 1);
    const long long above = roots_at_least(g, NE_BINOM_N + 1);
    const long long big = roots_at_least(g, std::max(NE_LIGHT_D + 1, need));
    const long long all = std::max(big, roots_at_least(g, need));
    const long long n_big = big - above;
    g->scratch_queue.ensure(256 + sizeof(unsigned int) * (size_t)std::max<long long>(n_big, 1));
    unsigned long long* tickets = g->scratch_queue.as<unsigned long long>();
    GPM_CUDA(cudaMemsetAsync(tickets, 0, 256 + sizeof(unsigned int) * (size_t)n_big, s));
    if (n_big > 0) {
        p.first = above;
        p.last = big;
        p.maxd = std::min(g->max_outdeg, NE_BINOM_N);
        p.w = (p.maxd + 31) / 32;
        p.ws = p.w | 1;
        const bool deep = k_hi >= 5;
        // A child's set has fewer members than its root's list: lists well above
        // NE_DIRECT_M, or an eighth of them above it (complete multipartite graphs and
        // G(n, 0.5 .. 0.95) of 250 to 1,200 vertices: 0.37 to 0.78; the core of the
        // Chung-Lu graph of 10^6: 0.08, lists of up to 297).
        const bool direct = deep && (g->max_outdeg > 2 * NE_DIRECT_M ||
                                     8 * (roots_at_least(g, NE_DIRECT_M + 1) - above) >= n_big);
        const void* heavy = !deep ? (const void*)k_clique_ne_heavy<false, false>
                            : direct ? (const void*)k_clique_ne_heavy<true, true> : (const void*)k_clique_ne_heavy<true, false>;
        p.warp_words = ne_warp_words(p.maxd, p.w, deep);
        p.n_help = std::max(0ll, roots_at_least(g, NE_HELP_D + 1) - above);
        p.rounds = k_hi >= 6 ? NE_HELP_ROUNDS : 0;
        p.grab = k_hi >= 6 ? 2 : 16;
        p.ticket = tickets;
        p.next_child = reinterpret_cast<unsigned int*>(tickets + 32);
        const size_t smem = 4 * ((size_t)ne_block_words(p.maxd, p.ws) + (size_t)NE_WARPS * p.warp_words);
        allow_shared(heavy, smem);
        Grid gr = plan_grid(g, heavy, NE_WARPS, smem);
        gr.blocks = (int)std::min<long long>(gr.blocks, n_big + p.n_help * p.rounds);
        p.busy = made.add(ctl, gr);
        if (!deep) k_clique_ne_heavy<false, false><<<gr.blocks, NE_WARPS * 32, smem, s>>>(p);
        else if (direct) k_clique_ne_heavy<true, true><<<gr.blocks, NE_WARPS * 32, smem, s>>>(p);
        else k_clique_ne_heavy<true, false><<<gr.blocks, NE_WARPS * 32, smem, s>>>(p);
        GPM_CUDA(cudaGetLastError());
    }
    if (all > big) {
        p.first = big;
        p.last = all;
        p.ticket = tickets + 16;
        const long long want = (all - big + NE_LIGHT_GRAB * NE_LIGHT_WARPS - 1) / (NE_LIGHT_GRAB * NE_LIGHT_WARPS);
        Grid gr = plan_grid(g, (const void*)k_clique_ne_light, NE_LIGHT_WARPS, 0);
        gr.blocks = (int)std::min<long long>(want, gr.blocks);
        p.busy = made.add(ctl, gr);
        k_clique_ne_light<<<gr.blocks, NE_LIGHT_WARPS * 32, 0, s>>>(p);
        GPM_CUDA(cudaGetLastError());
    }
}

}  // namespace gpm
