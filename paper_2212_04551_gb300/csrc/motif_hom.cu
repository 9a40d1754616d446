// motif_hom.cu -- whole-graph induced motif counts, k = 3 .. 5, from
// homomorphism counts (the result of Algorithm 4, motif counting, without
// visiting the k-vertex sets).
//
// The number of induced copies of a connected pattern P is a fixed integer
// combination of the numbers of homomorphisms into G of the connected graphs
// on at most k vertices (31 for k = 5): inclusion-exclusion over the edges
// that P lacks gives the injective ones, Moebius inversion over the partitions
// of the vertices (blocks without inner edges) the homomorphisms.  The
// combination is computed once per k on the host (hom_table).
//
// Every one of these numbers is a sum over the vertices u of what one warp
// finds around u, with c(w) the common neighbours of u and w (two-step walks),
// t = c on the neighbours of u, and L the graph among the neighbours of u
// (bit rows in shared memory):
//
//   * c from the adjacency lists of N(u); cycles of four sum c^2, K_{2,3} c^3,
//     and the patterns grown on the edge u-v by triangles t, t^2, t^3;
//   * K4, K5, wheel, gem and their relatives from pairs of rows of L;
//   * houses from the sums of c over the lists of N(u), cycles of five from the
//     sum of c(w) c(x) over the edges of the graph, the wheel without a spoke
//     from the edges of L inside N(w), w with c(w) >= 2.
//
// The work is a few scans of the lists around u, where the walk scans them for
// every (k-2)-set.  Everything the scans look up lies in shared
// memory, so the rule hom_applies() asks for graphs whose arrays fit: at most
// 2^14 vertices and degrees up to 2^10, which bounds every homomorphism count
// (n d^(k-1)) by 2^54, so that 64-bit sums are exact.
//
// What bounds it: the latency of the loads and lookups (one warp per vertex;
// issue slots 0.3 busy), hence several entries per lane in flight in every scan.
// The warps in flight are limited by their arrays in shared memory, 8 bytes per
// vertex of the graph and the rows: 8 warps per SM on the block-model graph of
// 2,000 vertices (21.7 KB each), 1 at 2^14; on small graphs by the 128
// registers of k = 5 (16).
// Measured, whole call, the walk / this: G(516, 1200) k = 4 857 / 33 us;
// block-model graph of 2,000 vertices k = 5 199 / 1.4 ms; 4,096 small graphs,
// 4-cliques and 5-motifs 150 / 6.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "common.cuh"
#include "motif_hom.cuh"

namespace gpm {

// Exponents (d, s, T) of the H_UNIFORM sums, in their order.
__device__ __constant__ static unsigned char kHomExp[H_UNIFORM][3] = {
    {0, 0, 0}, {1, 0, 0}, {2, 0, 0}, {0, 0, 1}, {3, 0, 0}, {1, 1, 0}, {1, 0, 1},
    {4, 0, 0}, {0, 2, 0}, {2, 1, 0}, {2, 0, 1}, {0, 1, 1}, {0, 0, 2}};

// One warp's shared arrays.
struct HomWarp {
    uint32_t* c;       // per vertex: two-step walks from u (d <= 32: the set of places in N(u) they pass)
    uint16_t* idx;     // per vertex: its place in N(u), from 1 (0: not in N(u))
    uint16_t* seen;    // the vertices with c > 0
    int* t;            // per neighbour: triangles on its edge to u
    int* at;           // per neighbour: where its list begins (later: how far it has been read) ...
    int* end;          // ... and ends
    uint32_t* L;       // bit rows of the graph on N(u)
    uint32_t* M;       // bit sets over N(u), of a range of vertices
};

// Lane-private sums, zeroed at every change of the graph.
struct HomSums {
    unsigned long long v[HOM_N];   // (indexed by constants only: registers)
};

template <int K>
__device__ __forceinline__ void hom_flush(const HomLaunch& p, HomSums& a, unsigned long long& uniform, int g, int lane) {
    unsigned long long mine = uniform;
#pragma unroll
    for (int j = H_UNIFORM; j < HOM_N; j++) {
        const unsigned long long x = gpm_warp_sum(a.v[j]);
        if (lane == j) mine = x;
        a.v[j] = 0;
    }
    if (lane < HOM_N && mine) atomicAdd(&p.hom[(long long)g * HOM_N + lane], mine);
    uniform = 0;
}

// Part `part` of p.parts of the vertex u of the graph of vertices base .. last-1:
// all parts set up the arrays, and take turns at the loops over pairs of
// neighbours and over the lists two steps away; part 0 adds the other sums.
//
// With d <= 32 the walks to a vertex are kept as the set of neighbours they
// pass, one word: its population is c, at a neighbour it is the row of L, and
// the edges of L inside it need no scan.
template <int K>
__device__ __forceinline__ void hom_vertex(const HomLaunch& p, const HomWarp& k, HomSums& a,
                                           unsigned long long& uniform, unsigned long long& scanned, int u, int part,
                                           int base, int last, int lane) {
    const int beg = p.indptr[u], d = p.indptr[u + 1] - beg;
    const int32_t* N = p.indices + beg;
    const int w = (d + 31) >> 5, ws = w | 1;
    const int sub = lane & 7, grp = lane >> 3;
    const bool sets = K >= 4 && d <= 32;           // warp-uniform
    // ---- N(u): places, degrees; clear the rows
    unsigned s = 0;
    for (int i = lane; i < d; i += 32) {
        const int v = N[i];
        const int b = p.indptr[v], e = p.indptr[v + 1];
        k.idx[v - base] = (uint16_t)(i + 1);
        k.at[i] = b;
        k.end[i] = e;
        s += (unsigned)(e - b);
    }
    s = __reduce_add_sync(GPM_FULL_MASK, s);
    if (K >= 4 && !sets)
        for (int i = lane; i < d * ws; i += 32) k.L[i] = 0u;
    __syncwarp();
    // ---- the lists of N(u), eight lanes each: c, the rows of L
    int n_seen = 0;
    unsigned T = 0;                                // lane's entries inside N(u)
    for (int i0 = 0; i0 < d; i0 += 4) {
        const int i = i0 + grp;
        int b = 0, e = 0;
        if (i < d) {
            b = k.at[i];
            e = k.end[i];
        }
        // (two entries per lane in flight)
        for (int q = b + sub; __any_sync(GPM_FULL_MASK, q < e); q += 16) {
            int xs[2];
#pragma unroll
            for (int z = 0; z < 2; z++) xs[z] = q + 8 * z < e ? p.indices[q + 8 * z] - base : -1;
#pragma unroll
            for (int z = 0; z < 2; z++) {
                const int x = xs[z];
                bool fresh = false;
                if (x >= 0) {
                    if (sets) {
                        fresh = atomicOr(&k.c[x], 1u << i) == 0u;
                    } else {
                        const int j = k.idx[x];
                        if (j) {
                            T++;
                            if (K >= 4) atomicOr(&k.L[i * ws + ((j - 1) >> 5)], 1u << ((j - 1) & 31));
                        }
                        if (K >= 4) fresh = atomicAdd(&k.c[x], 1u) == 0u;
                    }
                }
                if (K >= 4) {
                    const unsigned bal = __ballot_sync(GPM_FULL_MASK, fresh);
                    if (fresh) k.seen[n_seen + __popc(bal & gpm_lanemask_lt())] = (uint16_t)x;
                    n_seen += __popc(bal);
                }
            }
        }
    }
    __syncwarp();
    if (sets && lane < d) {
        const uint32_t row = k.c[N[lane] - base];
        k.L[lane] = row;
        T = __popc(row);
    }
    T = __reduce_add_sync(GPM_FULL_MASK, T);
    __syncwarp();
    if (lane == 0) scanned += s;
    // ---- d^a s^b T^c: lane j holds the j-th such sum
    if (part == 0 && lane < H_UNIFORM) {
        unsigned long long x = 1;
        for (int q = kHomExp[lane][0]; q > 0; q--) x *= (unsigned)d;
        for (int q = kHomExp[lane][1]; q > 0; q--) x *= s;
        for (int q = kHomExp[lane][2]; q > 0; q--) x *= T;
        uniform += x;
    }
    const unsigned long long ud = (unsigned)d;
    if (K >= 4) {
        // ---- sums over the two-step walks
        if (part == 0) {
            unsigned long long c2 = 0;
            for (int i = lane; i < n_seen; i += 32) {
                const uint32_t m = k.c[k.seen[i]];
                const unsigned long long c = sets ? __popc(m) : m;
                c2 += c * c;
                if (K == 5) {
                    a.v[H_K23] += c * c * c;
                    if (sets && c >= 2 && T) {         // edges of L in N(w), both directions
                        unsigned inside = 0;
                        for (uint32_t y = m; y; y &= y - 1u) inside += __popc(k.L[__ffs(y) - 1] & m);
                        a.v[H_SPOKE] += c * inside;
                    }
                }
            }
            a.v[H_CYCLE4] += c2;
            if (K == 5) a.v[H_BANNER] += c2 * ud;
        }
        // ---- sums over the edges u-v
        for (int i = lane; i < d; i += 32) {
            const uint32_t m = k.c[N[i] - base];
            const unsigned long long t = sets ? __popc(m) : m;
            k.t[i] = (int)t;
            if (part) continue;
            a.v[H_DIAMOND] += t * t;
            if (K == 5) {
                a.v[H_BULL] += t * ud * (unsigned)(k.end[i] - k.at[i]);
                a.v[H_DART] += t * t * ud;
                a.v[H_BOOK] += t * t * t;
                a.v[H_WHEEL] += t * t;             // a pair (i, i) below
            }
        }
        __syncwarp();
    }
    // ---- pairs of neighbours i < j
    if (K >= 4 && T) {
        unsigned long long k4 = 0;
        auto pair = [&](int i, int j) {
            const uint32_t* ri = k.L + i * ws;
            const uint32_t* rj = k.L + j * ws;
            unsigned cl = 0;
            for (int z = 0; z < w; z++) cl += __popc(ri[z] & rj[z]);
            const bool adj = (ri[j >> 5] >> (j & 31)) & 1u;
            if (K == 5) a.v[H_WHEEL] += 2ull * cl * cl;
            if (!adj) return;
            k4 += 2 * cl;
            if (K == 5) {
                const int ti = k.t[i], tj = k.t[j];
                a.v[H_K5E] += 2ull * cl * cl;
                a.v[H_GEM] += 2ull * (unsigned)ti * (unsigned)tj;
                a.v[H_KITE] += (unsigned long long)ti * (unsigned)(k.end[j] - k.at[j]) +
                               (unsigned long long)tj * (unsigned)(k.end[i] - k.at[i]);
                a.v[H_K5P3] += (unsigned long long)(ti + tj) * cl;
                // 4-cliques of L with lowest places i, j
                unsigned q5 = 0;
                for (int z = j >> 5; z < w; z++) {
                    uint32_t y = ri[z] & rj[z];
                    if (z == (j >> 5)) y &= 0xfffffffeu << (j & 31);
                    while (y) {
                        const uint32_t* ry = k.L + (32 * z + __ffs(y) - 1) * ws;
                        y &= y - 1u;
                        q5 += __popc(y & ry[z]);
                        for (int o = z + 1; o < w; o++) q5 += __popc(ri[o] & rj[o] & ry[o]);
                    }
                }
                a.v[H_K5] += 24ull * q5;
            }
        };
        if (sets) {
            // (few neighbours: all pairs in one range, numbered j (j - 1) / 2 + i)
            for (int t = 32 * part + lane; t < d * (d - 1) / 2; t += 32 * p.parts) {
                int j = (int)(0.5f + sqrtf(0.25f + 2.f * (float)t));
                if (j * (j - 1) / 2 > t) j--;
                if (j * (j + 1) / 2 <= t) j++;
                pair(t - j * (j - 1) / 2, j);
            }
        } else {
            for (int i = part; i < d; i += p.parts) {
                if (!k.t[i]) continue;                 // warp-uniform: an empty row
                for (int j = i + 1 + lane; j < d; j += 32) pair(i, j);
            }
        }
        a.v[H_K4] += k4;
        if (K == 5) a.v[H_K4TAIL] += k4 * ud;
    }
    if (K == 5) {
        // ---- houses: the lists of N(u) once more, now that c is known
        for (int i0 = 4 * part; i0 < d; i0 += 4 * p.parts) {
            const int i = i0 + grp;
            if (i >= d || !k.t[i]) continue;
            unsigned long long y = 0;
            for (int q = k.at[i] + sub, e = k.end[i]; q < e; q += 16) {
                const int x0 = p.indices[q], x1 = q + 8 < e ? p.indices[q + 8] : -1;
                const uint32_t m0 = k.c[x0 - base], m1 = x1 >= 0 ? k.c[x1 - base] : 0u;
                y += sets ? __popc(m0) + __popc(m1) : m0 + m1;
            }
            a.v[H_HOUSE] += (unsigned)k.t[i] * y;
        }
        // ---- cycles of five: sum of c(w) c(x) over the edges w - x, from the
        // lists of all w with c(w) > 0, or, when these hold more than an eighth
        // of the graph, from its edge list (one load and two lookups per edge)
        unsigned near = 0;
        for (int i = lane; i < n_seen; i += 32) near += (unsigned)p.deg[base + k.seen[i]];
        near = __reduce_add_sync(GPM_FULL_MASK, near);
        const int eb = p.indptr[base], ee = p.indptr[last];
        unsigned long long c5 = 0;
        if (8ll * near >= ee - eb) {
            // (four edges per lane in flight: the loads' latency is the loop's time)
            const int step = 32 * p.parts;
            int q = eb + 32 * part + lane;
            for (; q + 3 * step < ee; q += 4 * step) {
                uint32_t wx[4];
#pragma unroll
                for (int z = 0; z < 4; z++) wx[z] = p.edges[q + z * step];
#pragma unroll
                for (int z = 0; z < 4; z++) {
                    const uint32_t cw = k.c[wx[z] >> 16], cx = k.c[wx[z] & 0xffffu];
                    c5 += sets ? (unsigned)(__popc(cw) * __popc(cx)) : (unsigned long long)cw * cx;
                }
            }
            for (; q < ee; q += step) {
                const uint32_t wx = p.edges[q];
                const uint32_t cw = k.c[wx >> 16], cx = k.c[wx & 0xffffu];
                c5 += sets ? (unsigned)(__popc(cw) * __popc(cx)) : (unsigned long long)cw * cx;
            }
        } else {
            for (int i0 = 4 * part; i0 < n_seen; i0 += 4 * p.parts) {
                if (i0 + grp >= n_seen) continue;
                const int x = k.seen[i0 + grp];
                const uint32_t m = k.c[x];
                unsigned long long y = 0;
                for (int q = p.indptr[base + x] + sub, e = p.indptr[base + x + 1]; q < e; q += 8) {
                    const uint32_t mz = k.c[p.indices[q] - base];
                    y += sets ? __popc(mz) : mz;
                }
                c5 += (sets ? __popc(m) : m) * y;
            }
        }
        a.v[H_CYCLE5] += c5;
        // ---- the edges of L inside N(w), d > 32: the sets N(w) n N(u) of a range
        // of vertices w at a time, filled from the lists of N(u) (sorted: each
        // goes on where the last range ended)
        if (!sets && T) {
            const int span = p.m_words / w;            // vertices per range
            const int from = (int)((long long)(last - base) * part / p.parts);
            const int upto = (int)((long long)(last - base) * (part + 1) / p.parts);
            for (int i = lane; i < d; i += 32) {       // first neighbour of N[i] in this part's range
                int b = k.at[i], e = k.end[i];
                while (b < e) {
                    const int mid = (b + e) >> 1;
                    if (p.indices[mid] - base < from) b = mid + 1; else e = mid;
                }
                k.at[i] = b;
            }
            __syncwarp();
            for (int lo = from; lo < upto; lo += span) {
                const int hi = min(lo + span, upto);
                for (int z = lane; z < (hi - lo) * w; z += 32) k.M[z] = 0u;
                __syncwarp();
                for (int i0 = 0; i0 < d; i0 += 4) {
                    const int i = i0 + grp;
                    int q = 0, e = 0;
                    if (i < d) {
                        q = k.at[i] + sub;
                        e = k.end[i];
                    }
                    __syncwarp();                      // at[i] is read by its eight lanes
                    int done = 0;
                    for (; q < e; q += 8) {
                        const int x = p.indices[q] - base;
                        // (x < lo: only in an unchecked graph, whose lists may not be sorted)
                        if ((unsigned)(x - lo) >= (unsigned)(hi - lo)) break;
                        atomicOr(&k.M[(x - lo) * w + (i >> 5)], 1u << (i & 31));
                        done++;
                    }
                    if (i < d && done) atomicAdd(&k.at[i], done);
                }
                __syncwarp();
                for (int x = lo + lane; x < hi; x += 32) {
                    const unsigned c = k.c[x];
                    if (c < 2) continue;
                    const uint32_t* M = k.M + (x - lo) * w;
                    unsigned inside = 0;               // both directions
                    for (int z = 0; z < w; z++)
                        for (uint32_t y = M[z]; y; y &= y - 1u) {
                            const uint32_t* r = k.L + (32 * z + __ffs(y) - 1) * ws;
                            for (int o = 0; o < w; o++) inside += __popc(r[o] & M[o]);
                        }
                    a.v[H_SPOKE] += (unsigned long long)c * inside;
                }
                __syncwarp();
            }
        }
    }
    // ---- clear what was touched (no lane reads it any more)
    __syncwarp();
    for (int i = lane; i < n_seen; i += 32) k.c[k.seen[i]] = 0u;
    for (int i = lane; i < d; i += 32) k.idx[N[i] - base] = 0;
    __syncwarp();
}

template <int K>
__global__ void __launch_bounds__(HOM_WARPS * 32, K == 5 ? 4 : 8) k_hom(HomLaunch p) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31;
    uint32_t* mine = smem + (threadIdx.x >> 5) * p.warp_words;
    const int n4 = (p.maxn + 3) & ~3, d4 = (p.maxd + 3) & ~3, w = (p.maxd + 31) >> 5;
    HomWarp k;
    k.idx = reinterpret_cast<uint16_t*>(mine);
    k.seen = k.idx + n4;
    k.c = mine + n4;
    k.t = reinterpret_cast<int*>(k.c + n4);
    k.at = K == 3 ? reinterpret_cast<int*>(mine + n4 / 2) : k.t + d4;     // (k = 3: idx, at and end only)
    k.end = k.at + d4;
    k.L = reinterpret_cast<uint32_t*>(k.end + d4);
    k.M = k.L + p.maxd * (w | 1);
    for (int i = lane; i < (K == 3 ? n4 / 2 : 2 * n4); i += 32) mine[i] = 0u;
    __syncwarp();
    HomSums a;
#pragma unroll
    for (int j = 0; j < HOM_N; j++) a.v[j] = 0;
    unsigned long long uniform = 0, scanned = 0, units = 0;
    const unsigned long long t0 = gpm_globaltimer();
    int g = -1, base = 0, last = 0;
    for (;;) {
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(p.ticket, (unsigned long long)p.grab);
        at = __shfl_sync(GPM_FULL_MASK, at, 0);
        if (at >= (unsigned long long)(p.n * p.parts)) break;
        const long long upto = min((long long)at + p.grab, p.n * p.parts);
        for (long long i = (long long)at; i < upto; i++) {
            const int u = (int)(i / p.parts), part = (int)(i % p.parts);
            const int gu = p.vgraph ? p.vgraph[u] : 0;
            if (gu != g) {
                if (g >= 0) hom_flush<K>(p, a, uniform, g, lane);
                g = gu;
                base = p.goff ? p.goff[gu] : 0;
                last = p.goff ? p.goff[gu + 1] : (int)p.n;
            }
            hom_vertex<K>(p, k, a, uniform, scanned, u, part, base, last, lane);
            units += part == 0;
        }
    }
    if (g >= 0) hom_flush<K>(p, a, uniform, g, lane);
    scanned = gpm_warp_sum(scanned);
    if (lane == 0) {
        atomicAdd(&p.ctl->units_done, units);
        atomicAdd(&p.ctl->word_ops, scanned);
        atomicAdd(p.busy, gpm_globaltimer() - t0);
    }
}

// per adjacency entry, its two ends within their graph: (vertex << 16) | neighbour
__global__ void k_hom_edges(const int32_t* __restrict__ indptr, const int32_t* __restrict__ indices,
                            const int32_t* __restrict__ goff, const int32_t* __restrict__ vgraph, int32_t n,
                            uint32_t* __restrict__ edges) {
    for (long long v = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 3; v < n;
         v += ((long long)gridDim.x * blockDim.x) >> 3) {
        const int base = vgraph ? goff[vgraph[v]] : 0;
        for (int q = indptr[v] + (threadIdx.x & 7), e = indptr[v + 1]; q < e; q += 8)
            edges[q] = (uint32_t)(v - base) << 16 | (uint32_t)(indices[q] - base);
    }
}

// thread per (graph, pattern)
__global__ void k_hom_finish(const unsigned long long* __restrict__ hom, long long n_out, int npat,
                             const long long* __restrict__ coef, unsigned long long* __restrict__ out, int clique_hom,
                             int clique_aut, unsigned long long* __restrict__ clique_out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_out; i += (long long)gridDim.x * blockDim.x) {
        const long long g = i / npat, pat = i % npat;
        const unsigned long long* h = hom + g * HOM_N;
        unsigned long long sum = 0;
        for (int j = 0; j < HOM_N; j++) sum += (unsigned long long)coef[pat * HOM_N + j] * h[j];
        out[i] = sum / (unsigned long long)coef[(long long)npat * HOM_N + pat];
        if (clique_out && pat == 0) clique_out[g] = h[clique_hom] / (unsigned)clique_aut;
    }
}

// ------------------------------------------------------------------- host

bool hom_applies(long long n, long long d, int k) {
    if (k < 3 || k > 5 || n < 1 || n > HOM_MAX_N || d > HOM_MAX_D) return false;
    return sizeof(uint32_t) * (size_t)hom_warp_words((int)n, (int)d, k) <= 220 * 1024;
}

// words of the bit sets of a range of vertices (d > 32): 4 KB, at least one set, at most all
int hom_m_words(int n, int d) {
    const int w = (d + 31) >> 5;
    return d <= 32 ? 0 : std::min(std::max(1024, w), n * w);
}

int hom_warp_words(int n, int d, int k) {
    const int n4 = (n + 3) & ~3, d4 = (d + 3) & ~3, w = (d + 31) >> 5;
    if (k == 3) return n4 / 2 + 2 * d4;                  // (idx, at and end only)
    return 2 * n4 + 3 * d4 + ((d * (w | 1) + (k == 5 ? hom_m_words(n, d) : 0) + 3) & ~3);
}

static const void* hom_kernel(int k) {
    return k == 3 ? (const void*)k_hom<3> : k == 4 ? (const void*)k_hom<4> : (const void*)k_hom<5>;
}

const uint32_t* ensure_hom_edges(gpm_graph* g, const int32_t* goff, const int32_t* vgraph) {
    if (!g->hom_edges.ptr) {
        DevBuf e;
        e.ensure(sizeof(uint32_t) * (size_t)std::max<int64_t>(g->nnz, 1));
        if (g->n > 0)
            k_hom_edges<<<std::max(1, std::min((g->n + 31) / 32, g->num_sms * 8)), 256, 0, g->stream>>>(
                g->indptr.as<int32_t>(), g->indices.as<int32_t>(), goff, vgraph, g->n, e.as<uint32_t>());
        GPM_CUDA(cudaGetLastError());
        g->hom_edges = std::move(e);
    }
    return g->hom_edges.as<uint32_t>();
}

Grid plan_hom(HomLaunch& p, int k, int sms, const gpm_config& cfg) {
    p.warp_words = hom_warp_words(p.maxn, p.maxd, k);
    p.m_words = hom_m_words(p.maxn, p.maxd);
    Grid gr;
    gr.warps_per_block = cfg.warps_per_block > 0 ? std::min(cfg.warps_per_block, HOM_WARPS) : HOM_WARPS;
    while (gr.warps_per_block > 1 && 4 * (size_t)p.warp_words * gr.warps_per_block > 220 * 1024) gr.warps_per_block /= 2;
    const size_t smem = 4 * (size_t)p.warp_words * gr.warps_per_block;
    allow_shared(hom_kernel(k), smem);
    long long per_sm = std::max(1, resident_blocks(hom_kernel(k), gr.warps_per_block * 32, smem));
    if (cfg.blocks_per_sm > 0) per_sm = std::min<long long>(per_sm, cfg.blocks_per_sm);
    // k = 5, few vertices: each is shared by several warps, so that the last
    // round of vertices is not a whole vertex long (block-model graph of 2,000
    // vertices on 1,824 warps)
    p.parts = k < 5 || p.vgraph ? 1 : (int)std::max(1ll, std::min(16ll, 8 * per_sm * sms * gr.warps_per_block / p.n));
    const long long tasks = (p.n * p.parts + p.grab - 1) / p.grab;
    gr.blocks = (int)std::min<long long>(per_sm * sms, (tasks + gr.warps_per_block - 1) / gr.warps_per_block);
    return gr;
}

cudaError_t launch_hom(const HomLaunch& p, int k, const Grid& gr, cudaStream_t s) {
    if (gr.blocks <= 0) return cudaSuccess;
    HomLaunch q = p;
    void* args[] = {&q};
    return cudaLaunchKernel(hom_kernel(k), dim3(gr.blocks), dim3(gr.warps_per_block * 32), args,
                            4 * (size_t)p.warp_words * gr.warps_per_block, s);
}

void run_motif_hom(gpm_graph* g, int k, uint64_t* counts_out) {
    const HomTable& t = hom_table(k);
    cudaStream_t s = g->stream;
    struct Result {
        Control ctl;
        unsigned long long hom[HOM_N];
    };
    g->scratch_small.ensure(sizeof(Result));
    Result* r = g->scratch_small.as<Result>();
    GPM_CUDA(cudaMemsetAsync(r, 0, sizeof(Result), s));
    HomLaunch p{};
    p.indptr = g->indptr.as<int32_t>();
    p.indices = g->indices.as<int32_t>();
    p.deg = g->degree.as<int32_t>();
    p.n = p.maxn = g->n;
    p.maxd = std::max(g->max_deg, 1);
    p.grab = 1;
    p.hom = r->hom;
    p.ticket = &r->ctl.next_root;
    p.ctl = &r->ctl;
    p.busy = &r->ctl.busy_ns;
    if (k == 5) p.edges = ensure_hom_edges(g, nullptr, nullptr);
    const Grid gr = plan_hom(p, k, g->num_sms, g->cfg);
    GPM_CUDA(cudaEventRecord(g->ev0, s));
    GPM_CUDA(launch_hom(p, k, gr, s));
    GPM_CUDA(cudaEventRecord(g->ev1, s));
    Result h;
    GPM_CUDA(cudaMemcpyAsync(&h, r, sizeof(Result), cudaMemcpyDeviceToHost, s));
    GPM_CUDA(cudaStreamSynchronize(s));
    float ms = 0.f;
    GPM_CUDA(cudaEventElapsedTime(&ms, g->ev0, g->ev1));
    gpm_stats st{};
    st.kernel_ms = ms;
    st.units_done = h.ctl.units_done;
    st.word_ops = h.ctl.word_ops;
    st.busy_warp_ns = h.ctl.busy_ns;
    st.kernel_launches = 1;
    st.grid_blocks = gr.blocks;
    st.warps_per_block = gr.warps_per_block;
    g->stats = st;
    hom_combine(t, h.hom, counts_out);
}

void hom_combine(const HomTable& t, const unsigned long long* hom, uint64_t* counts_out) {
    for (int q = 0; q < t.npat; q++) {
        unsigned long long sum = 0;
        for (int j = 0; j < HOM_N; j++) sum += (unsigned long long)t.coef[(size_t)q * HOM_N + j] * hom[j];
        counts_out[q] = sum / (unsigned long long)t.aut[q];
    }
}

cudaError_t launch_hom_finish(const unsigned long long* hom, int n_graphs, int k, unsigned long long* out, int clique_k,
                              unsigned long long* clique_out, cudaStream_t s) {
    const int npat = hom_table(k).npat;
    const long long n_out = (long long)n_graphs * npat;
    if (n_out <= 0) return cudaSuccess;
    const long long* coef = device_hom_table(k, s);
    const int clique_hom = clique_k == 3 ? H_TRI : clique_k == 4 ? H_K4 : H_K5;
    const int clique_aut = clique_k == 3 ? 6 : clique_k == 4 ? 24 : 120;      // every clique is hit k! times
    k_hom_finish<<<(int)std::min<long long>((n_out + 255) / 256, 1024), 256, 0, s>>>(
        hom, n_out, npat, coef, out, clique_hom, clique_aut, clique_k > 0 ? clique_out : nullptr);
    return cudaGetLastError();
}

// ---- the combination of homomorphism counts

// Edges of each graph of Hom (vertices 0 ..), in the enum's order.
static const std::vector<std::vector<std::pair<int, int>>>& hom_edges() {
    static const std::vector<std::vector<std::pair<int, int>>> e = {
        {},                                                        // H_POINT
        {{0, 1}},                                                  // H_EDGE
        {{0, 1}, {0, 2}},                                          // H_CHERRY
        {{0, 1}, {0, 2}, {1, 2}},                                  // H_TRI
        {{0, 1}, {0, 2}, {0, 3}},                                  // H_STAR3
        {{0, 1}, {1, 2}, {2, 3}},                                  // H_PATH4
        {{0, 1}, {1, 2}, {0, 2}, {0, 3}},                          // H_PAW
        {{0, 1}, {0, 2}, {0, 3}, {0, 4}},                          // H_STAR4
        {{0, 1}, {1, 2}, {2, 3}, {3, 4}},                          // H_PATH5
        {{0, 1}, {0, 2}, {0, 3}, {3, 4}},                          // H_FORK
        {{0, 1}, {1, 2}, {0, 2}, {0, 3}, {0, 4}},                  // H_CRICKET
        {{0, 1}, {1, 2}, {0, 2}, {0, 3}, {3, 4}},                  // H_LOLLI
        {{0, 1}, {1, 2}, {0, 2}, {0, 3}, {0, 4}, {3, 4}},          // H_BOWTIE
        {{0, 1}, {1, 2}, {2, 3}, {0, 3}},                          // H_CYCLE4
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}},                  // H_DIAMOND
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}},          // H_K4
        {{0, 1}, {1, 2}, {2, 3}, {3, 4}, {0, 4}},                  // H_CYCLE5
        {{0, 1}, {1, 2}, {2, 3}, {0, 3}, {0, 4}},                  // H_BANNER
        {{0, 1}, {1, 2}, {0, 2}, {0, 3}, {1, 4}},                  // H_BULL
        {{0, 2}, {0, 3}, {0, 4}, {1, 2}, {1, 3}, {1, 4}},          // H_K23
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {0, 4}},          // H_DART
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 4}},          // H_KITE
        {{0, 1}, {1, 2}, {2, 3}, {0, 3}, {0, 4}, {1, 4}},          // H_HOUSE
        {{0, 1}, {1, 2}, {2, 3}, {4, 0}, {4, 1}, {4, 2}, {4, 3}},  // H_GEM
        {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {1, 3}, {0, 4}, {1, 4}},  // H_BOOK
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}, {0, 4}},  // H_K4TAIL
        {{0, 1}, {1, 2}, {2, 3}, {0, 3}, {4, 0}, {4, 1}, {4, 2}},  // H_SPOKE
        {{0, 1}, {1, 2}, {2, 3}, {0, 3}, {4, 0}, {4, 1}, {4, 2}, {4, 3}},          // H_WHEEL
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}, {0, 4}, {1, 4}},          // H_K5P3
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}, {0, 4}, {1, 4}, {2, 4}},  // H_K5E
        {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}, {0, 4}, {1, 4}, {2, 4}, {3, 4}}};   // H_K5
    return e;
}

// full code (bit i(i-1)/2 + j: edge {j, i}, j < i) of adjacency rows over k vertices
static uint32_t code_of(const std::vector<uint32_t>& adj) {
    uint32_t c = 0;
    for (int i = 1; i < (int)adj.size(); i++)
        for (int j = 0; j < i; j++)
            if ((adj[i] >> j) & 1u) c |= 1u << (i * (i - 1) / 2 + j);
    return c;
}

static std::vector<uint32_t> rows_of(uint32_t code, int k) {
    std::vector<uint32_t> adj(k, 0u);
    for (int i = 1; i < k; i++)
        for (int j = 0; j < i; j++)
            if ((code >> (i * (i - 1) / 2 + j)) & 1u) {
                adj[i] |= 1u << j;
                adj[j] |= 1u << i;
            }
    return adj;
}

// smallest code over all relabellings, and how many relabellings keep the code
static std::pair<uint32_t, int> canonical(uint32_t code, int k) {
    const std::vector<uint32_t> adj = rows_of(code, k);
    std::vector<int> at(k);
    for (int i = 0; i < k; i++) at[i] = i;
    uint32_t best = ~0u;
    int same = 0;
    do {
        std::vector<uint32_t> im(k, 0u);
        for (int i = 0; i < k; i++)
            for (int j = 0; j < k; j++)
                if ((adj[i] >> j) & 1u) im[at[i]] |= 1u << at[j];
        const uint32_t c = code_of(im);
        best = std::min(best, c);
        same += c == code ? 1 : 0;
    } while (std::next_permutation(at.begin(), at.end()));
    return {best, same};
}

// hom indices by (vertices, canonical code)
static const std::map<std::pair<int, uint32_t>, int>& hom_index() {
    static const std::map<std::pair<int, uint32_t>, int> idx = [] {
        std::map<std::pair<int, uint32_t>, int> m;
        const auto& all = hom_edges();
        for (int j = 0; j < (int)all.size(); j++) {
            int k = 1;
            for (const auto& e : all[j]) k = std::max(k, std::max(e.first, e.second) + 1);
            std::vector<uint32_t> adj(k, 0u);
            for (const auto& e : all[j]) {
                adj[e.first] |= 1u << e.second;
                adj[e.second] |= 1u << e.first;
            }
            m[{k, canonical(code_of(adj), k).first}] = j;
        }
        return m;
    }();
    return idx;
}

// injective homomorphisms of a k-vertex graph: mu(partition) times the
// homomorphisms of the quotient, added to out[] with the factor f
static void add_injective(uint32_t code, int k, long long f, long long* out) {
    const std::vector<uint32_t> adj = rows_of(code, k);
    std::vector<int> block(k, 0);
    static const long long mu[6] = {1, 1, -1, 2, -6, 24};   // (-1)^(b-1) (b-1)! by block size
    auto visit = [&](auto&& self, int v, int blocks) -> void {
        if (v == k) {
            long long m = f;
            std::vector<uint32_t> mask(blocks, 0u), q(blocks, 0u);
            for (int i = 0; i < k; i++) mask[block[i]] |= 1u << i;
            for (int b = 0; b < blocks; b++) m *= mu[__builtin_popcount(mask[b])];
            for (int i = 0; i < k; i++)
                for (int j = 0; j < k; j++)
                    if ((adj[i] >> j) & 1u) q[block[i]] |= 1u << block[j];
            out[hom_index().at({blocks, canonical(code_of(q), blocks).first})] += m;
            return;
        }
        for (int b = 0; b <= blocks; b++) {
            bool free_of_edges = true;
            for (int i = 0; i < v; i++)
                if (block[i] == b && ((adj[v] >> i) & 1u)) free_of_edges = false;
            if (!free_of_edges) continue;
            block[v] = b;
            self(self, v + 1, std::max(blocks, b + 1));
        }
    };
    visit(visit, 0, 0);
}

const HomTable& hom_table(int k) {
    static std::mutex mu;
    static std::map<int, HomTable> tables;
    std::lock_guard<std::mutex> lock(mu);
    auto it = tables.find(k);
    if (it != tables.end()) return it->second;
    const PatternTable& pat = pattern_table(k);
    HomTable t;
    t.k = k;
    t.npat = (int)pat.num_patterns;
    t.coef.assign((size_t)t.npat * HOM_N, 0);
    t.aut.assign(t.npat, 1);
    const uint32_t full = (1u << (k * (k - 1) / 2)) - 1u;
    for (int p = 0; p < t.npat; p++) {
        const uint32_t code = (uint32_t)pat.pattern_code[p];
        t.aut[p] = canonical(code, k).second;
        // every graph on the same vertices with more edges, by inclusion-exclusion
        const uint32_t free_edges = full & ~code;
        for (uint32_t more = free_edges;; more = (more - 1) & free_edges) {
            add_injective(code | more, k, __builtin_popcount(more) & 1 ? -1 : 1, &t.coef[(size_t)p * HOM_N]);
            if (!more) break;
        }
    }
    return tables[k] = std::move(t);
}

const long long* device_hom_table(int k, cudaStream_t s) {
    static std::mutex mu;
    static std::map<std::pair<int, int>, long long*> tables;
    const HomTable& t = hom_table(k);
    int dev = 0;
    GPM_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    auto it = tables.find({dev, k});
    if (it != tables.end()) return it->second;
    std::vector<long long> both(t.coef);
    both.insert(both.end(), t.aut.begin(), t.aut.end());
    auto* d = static_cast<long long*>(upload_table(both.data(), both.size() * sizeof(both[0]), s, "homomorphism table"));
    return tables[{dev, k}] = d;
}

}  // namespace gpm
