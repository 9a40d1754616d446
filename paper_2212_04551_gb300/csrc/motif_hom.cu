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
//   * cycles of five, houses and the wheel without a spoke from one more scan,
//     of the lists of all w with c(w) > 0: y(w) = sum of c over N(w), and the
//     edges of L inside N(w).
//
// The work is one scan of the lists two steps away per vertex, where the walk
// scans them for every (k-2)-set.  Everything the scans look up lies in shared
// memory, so the rule hom_applies() asks for graphs whose arrays fit: at most
// 2^14 vertices and degrees up to 2^10, which bounds every homomorphism count
// (n d^(k-1)) by 2^54, so that 64-bit sums are exact.
//
// What bounds it: instruction issue and shared-memory latency of the scans
// (one warp per vertex, 16 warps per SM at 128 registers for k = 5).
// Measured, whole call: G(516, 1200) k = 4 857 -> 34 us; block-model graph of
// 2,000 vertices k = 5 199 -> 3.9 ms; 4,096 small graphs, 4-cliques and
// 5-motifs 150 -> 17.7 ms.
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
    uint32_t* c;       // per vertex: two-step walks from u
    uint16_t* idx;     // per vertex: its place in N(u), from 1 (0: not in N(u))
    uint16_t* seen;    // the vertices with c > 0
    int* t;            // per neighbour: triangles on its edge to u
    int* d;            // per neighbour: its degree
    uint32_t* L;       // bit rows of the graph on N(u)
    uint32_t* M;       // four bit sets over N(u)
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

// The vertex u of the graph whose first vertex is base.
template <int K>
__device__ __forceinline__ void hom_vertex(const HomLaunch& p, const HomWarp& k, HomSums& a,
                                           unsigned long long& uniform, unsigned long long& scanned, int u, int base,
                                           int lane) {
    const int beg = p.indptr[u], d = p.indptr[u + 1] - beg;
    const int32_t* N = p.indices + beg;
    const int w = (d + 31) >> 5, ws = w | 1;
    const int sub = lane & 7, grp = lane >> 3;
    // ---- N(u): places, degrees; clear the rows
    unsigned s = 0;
    for (int i = lane; i < d; i += 32) {
        const int v = N[i];
        const int dv = p.deg[v];
        k.idx[v - base] = (uint16_t)(i + 1);
        k.d[i] = dv;
        s += (unsigned)dv;
    }
    s = __reduce_add_sync(GPM_FULL_MASK, s);
    if (K >= 4)
        for (int i = lane; i < d * ws; i += 32) k.L[i] = 0u;
    __syncwarp();
    // ---- the lists of N(u), eight lanes each: c, the rows of L
    int n_seen = 0;
    unsigned T = 0;                                // lane's entries inside N(u)
    for (int i0 = 0; i0 < d; i0 += 4) {
        const int i = i0 + grp;
        int b = 0, e = 0;
        if (i < d) {
            const int v = N[i];
            b = p.indptr[v];
            e = p.indptr[v + 1];
        }
        for (int q = b + sub; __any_sync(GPM_FULL_MASK, q < e); q += 8) {
            bool fresh = false;
            int x = 0;
            if (q < e) {
                x = p.indices[q] - base;
                const int j = k.idx[x];
                if (j) {
                    T++;
                    if (K >= 4) atomicOr(&k.L[i * ws + ((j - 1) >> 5)], 1u << ((j - 1) & 31));
                }
                if (K >= 4) fresh = atomicAdd(&k.c[x], 1u) == 0u;
            }
            if (K >= 4) {
                const unsigned bal = __ballot_sync(GPM_FULL_MASK, fresh);
                if (fresh) k.seen[n_seen + __popc(bal & gpm_lanemask_lt())] = (uint16_t)x;
                n_seen += __popc(bal);
            }
        }
    }
    T = __reduce_add_sync(GPM_FULL_MASK, T);
    __syncwarp();
    if (lane == 0) scanned += s;
    // ---- d^a s^b T^c: lane j holds the j-th such sum
    if (lane < H_UNIFORM) {
        unsigned long long x = 1;
        for (int q = kHomExp[lane][0]; q > 0; q--) x *= (unsigned)d;
        for (int q = kHomExp[lane][1]; q > 0; q--) x *= s;
        for (int q = kHomExp[lane][2]; q > 0; q--) x *= T;
        uniform += x;
    }
    const unsigned long long ud = (unsigned)d;
    if (K >= 4) {
        // ---- sums over the two-step walks
        unsigned long long c2 = 0;
        for (int i = lane; i < n_seen; i += 32) {
            const unsigned long long c = k.c[k.seen[i]];
            c2 += c * c;
            if (K == 5) a.v[H_K23] += c * c * c;
        }
        a.v[H_CYCLE4] += c2;
        if (K == 5) a.v[H_BANNER] += c2 * ud;
        // ---- sums over the edges u-v
        for (int i = lane; i < d; i += 32) {
            const unsigned long long t = k.c[N[i] - base];
            k.t[i] = (int)t;
            a.v[H_DIAMOND] += t * t;
            if (K == 5) {
                a.v[H_BULL] += t * ud * (unsigned)k.d[i];
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
        for (int i = 0; i < d; i++) {
            const int ti = k.t[i];
            if (!ti) continue;                     // warp-uniform: an empty row
            const uint32_t* ri = k.L + i * ws;
            const int di = k.d[i];
            for (int j = i + 1 + lane; j < d; j += 32) {
                const uint32_t* rj = k.L + j * ws;
                unsigned cl = 0;
                for (int z = 0; z < w; z++) cl += __popc(ri[z] & rj[z]);
                const bool adj = (ri[j >> 5] >> (j & 31)) & 1u;
                if (K == 5) a.v[H_WHEEL] += 2ull * cl * cl;
                if (!adj) continue;
                k4 += 2 * cl;
                if (K == 5) {
                    const int tj = k.t[j];
                    a.v[H_K5E] += 2ull * cl * cl;
                    a.v[H_GEM] += 2ull * (unsigned)ti * (unsigned)tj;
                    a.v[H_KITE] += (unsigned long long)ti * (unsigned)k.d[j] + (unsigned long long)tj * (unsigned)di;
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
            }
        }
        a.v[H_K4] += k4;
        if (K == 5) a.v[H_K4TAIL] += k4 * ud;
    }
    // ---- the lists of every w with c(w) > 0, eight lanes each
    if (K == 5) {
        for (int i0 = 0; i0 < n_seen; i0 += 4) {
            int x = -1, b = 0, e = 0;
            unsigned c = 0;
            if (i0 + grp < n_seen) {
                x = k.seen[i0 + grp];
                c = k.c[x];
                b = p.indptr[base + x];
                e = p.indptr[base + x + 1];
            }
            const bool rows = T && __any_sync(GPM_FULL_MASK, c >= 2);
            uint32_t* M = k.M + grp * w;
            if (rows) {
                for (int z = sub; z < w; z += 8) M[z] = 0u;
                __syncwarp();
            }
            unsigned long long y = 0;
            for (int q = b + sub; q < e; q += 8) {
                const int z = p.indices[q] - base;
                y += k.c[z];
                if (rows) {
                    const int j = k.idx[z];
                    if (j) atomicOr(&M[(j - 1) >> 5], 1u << ((j - 1) & 31));
                }
            }
            scanned += sub == 0 ? (unsigned)(e - b) : 0u;
            a.v[H_CYCLE5] += c * y;
            if (x >= 0 && k.idx[x]) a.v[H_HOUSE] += c * y;
            if (rows) {
                __syncwarp();
                unsigned inside = 0;               // edges of L in N(w), both directions
                if (c >= 2)
                    for (int j = sub; j < d; j += 8) {
                        if (!((M[j >> 5] >> (j & 31)) & 1u)) continue;
                        const uint32_t* rj = k.L + j * ws;
                        for (int z = 0; z < w; z++) inside += __popc(rj[z] & M[z]);
                    }
                a.v[H_SPOKE] += (unsigned long long)c * inside;
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
__global__ void __launch_bounds__(HOM_WARPS * 32) k_hom(HomLaunch p) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int lane = threadIdx.x & 31;
    uint32_t* mine = smem + (threadIdx.x >> 5) * p.warp_words;
    const int n4 = (p.maxn + 3) & ~3, d4 = (p.maxd + 3) & ~3, w = (p.maxd + 31) >> 5;
    HomWarp k;
    k.idx = reinterpret_cast<uint16_t*>(mine);
    k.seen = k.idx + n4;
    k.c = mine + n4;
    k.t = reinterpret_cast<int*>(k.c + n4);
    k.d = k.t + d4;
    k.L = reinterpret_cast<uint32_t*>(k.d + d4);
    k.M = k.L + p.maxd * (w | 1);
    for (int i = lane; i < (K == 3 ? n4 : 2 * n4); i += 32) mine[i] = 0u;
    __syncwarp();
    HomSums a;
#pragma unroll
    for (int j = 0; j < HOM_N; j++) a.v[j] = 0;
    unsigned long long uniform = 0, scanned = 0, units = 0;
    const unsigned long long t0 = gpm_globaltimer();
    int g = -1, base = 0;
    for (;;) {
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(p.ticket, (unsigned long long)p.grab);
        at = __shfl_sync(GPM_FULL_MASK, at, 0);
        if (at >= (unsigned long long)p.n) break;
        const long long upto = min((long long)at + p.grab, p.n);
        for (long long i = (long long)at; i < upto; i++) {
            const int u = p.order ? p.order[i] : (int)i;
            const int gu = p.vgraph ? p.vgraph[u] : 0;
            if (gu != g) {
                if (g >= 0) hom_flush<K>(p, a, uniform, g, lane);
                g = gu;
                base = p.goff ? p.goff[gu] : 0;
            }
            hom_vertex<K>(p, k, a, uniform, scanned, u, base, lane);
            units++;
        }
    }
    if (g >= 0) hom_flush<K>(p, a, uniform, g, lane);
    scanned = gpm_warp_sum(scanned);
    if (lane == 0) {
        atomicAdd(&p.ctl->units_done, units);
        atomicAdd(&p.ctl->word_ops, scanned);
        atomicAdd(&p.ctl->busy_ns, gpm_globaltimer() - t0);
    }
}

// thread per (graph, pattern)
__global__ void k_hom_finish(const unsigned long long* __restrict__ hom, long long n_out, int npat,
                             const long long* __restrict__ coef, unsigned long long* __restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_out; i += (long long)gridDim.x * blockDim.x) {
        const long long g = i / npat, pat = i % npat;
        const unsigned long long* h = hom + g * HOM_N;
        unsigned long long sum = 0;
        for (int j = 0; j < HOM_N; j++) sum += (unsigned long long)coef[pat * HOM_N + j] * h[j];
        out[i] = sum / (unsigned long long)coef[(long long)npat * HOM_N + pat];
    }
}

// ------------------------------------------------------------------- host

bool hom_applies(long long n, long long d, int k) {
    if (k < 3 || k > 5 || n < 1 || n > HOM_MAX_N || d > HOM_MAX_D) return false;
    return sizeof(uint32_t) * (size_t)hom_warp_words((int)n, (int)d, k) <= 220 * 1024;
}

int hom_warp_words(int n, int d, int k) {
    const int n4 = (n + 3) & ~3, d4 = (d + 3) & ~3, w = (d + 31) >> 5;
    if (k == 3) return n4 + n4 + 2 * d4;                 // (no rows)
    return 2 * n4 + 2 * d4 + ((d * (w | 1) + 4 * w + 3) & ~3);
}

static const void* hom_kernel(int k) {
    return k == 3 ? (const void*)k_hom<3> : k == 4 ? (const void*)k_hom<4> : (const void*)k_hom<5>;
}

Grid plan_hom(HomLaunch& p, int k, int sms) {
    p.warp_words = hom_warp_words(p.maxn, p.maxd, k);
    Grid gr;
    gr.warps_per_block = HOM_WARPS;
    while (gr.warps_per_block > 1 && 4 * (size_t)p.warp_words * gr.warps_per_block > 220 * 1024) gr.warps_per_block /= 2;
    const size_t smem = 4 * (size_t)p.warp_words * gr.warps_per_block;
    GPM_CUDA(cudaFuncSetAttribute(hom_kernel(k), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const long long per_sm = std::max(1, resident_blocks(hom_kernel(k), gr.warps_per_block * 32, smem));
    const long long tasks = (p.n + p.grab - 1) / p.grab;
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
    const Grid gr = plan_hom(p, k, g->num_sms);
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

cudaError_t launch_hom_finish(const unsigned long long* hom, int n_graphs, int k, unsigned long long* out, cudaStream_t s) {
    const int npat = hom_table(k).npat;
    const long long n_out = (long long)n_graphs * npat;
    if (n_out <= 0) return cudaSuccess;
    const long long* coef = device_hom_table(k);
    k_hom_finish<<<(int)std::min<long long>((n_out + 255) / 256, 1024), 256, 0, s>>>(hom, n_out, npat, coef, out);
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

const long long* device_hom_table(int k) {
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
    long long* d = nullptr;
    if (cudaMalloc(&d, both.size() * sizeof(long long)) != cudaSuccess) {
        cudaGetLastError();
        fail(GPM_ENOMEM, "cudaMalloc for the homomorphism table failed");
    }
    const cudaError_t e = cudaMemcpy(d, both.data(), both.size() * sizeof(long long), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(d);
        check_cuda(e, "cudaMemcpy(homomorphism table)");
    }
    return tables[{dev, k}] = d;
}

}  // namespace gpm
