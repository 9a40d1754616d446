// motif_sparse.cu -- whole-graph induced motif counts of 3 and 4 vertices on
// graphs too large for the per-vertex arrays of motif_hom.cu.
//
// The same combination of homomorphism counts (hom_table), from sums over the
// edges of the degree orientation instead of sums around every vertex:
//
//   * triangles, 4-cliques and the triangles t(e) of every edge come from the
//     row builds of the clique launch (clique_nonedge.cu), which meets each
//     triangle once;
//   * k_edge_sums adds up what degrees and t(e) decide: paths of four, paws
//     (t(e) (d_u + d_v)), diamonds (t(e)^2), stars;
//   * k_cycle4 counts the cycles of four at their last vertex u in the
//     (degree, id) order: with c(w) the paths u - v - w over v and w before u,
//     sum_w C(c(w), 2).  Only sum_v d(v) d+(v) paths are looked at (rmat16: 5.1e7,
//     where all paths of two edges are 4.0e8).  One block per u keeps c in shared
//     memory, as 16-bit counters, or in global memory when the graph has more
//     vertices than fit there; a second scan takes the counters out again.
//
// Bound: the random reads of degrees (L2) and the shared-memory atomics of
// k_cycle4, and the row builds.  Measured on rmat16 (65,536 vertices, 478 K
// edges), k = 4, whole call: the walk 202 ms, this 1.39 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "common.cuh"
#include "motif_hom.cuh"

namespace gpm {

constexpr int C4_THREADS = 1024;
constexpr int C4_SINGLE = 4096;               // the first positions are taken one by one, later ones in 32s
constexpr long long C4_SMEM_N = 110 * 1024;   // vertices whose 16-bit counters fit in shared memory

__global__ void k_edge_sums(const int32_t* __restrict__ off, const int32_t* __restrict__ adj,
                            const int32_t* __restrict__ outdeg, const int32_t* __restrict__ deg,
                            const unsigned int* __restrict__ tri, int32_t n, unsigned long long* __restrict__ hom,
                            unsigned long long* __restrict__ busy) {
    const unsigned long long t0 = gpm_globaltimer();
    __shared__ unsigned long long sum[5];
    if (threadIdx.x < 5) sum[threadIdx.x] = 0ull;
    __syncthreads();
    const int sub = threadIdx.x & 7;
    unsigned long long v[5] = {0, 0, 0, 0, 0};   // cherries, 3-stars, paths, paws, diamonds
    for (long long x = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 3; x < n;
         x += ((long long)gridDim.x * blockDim.x) >> 3) {
        const unsigned long long dx = (unsigned)deg[x];
        if (sub == 0) {
            v[0] += dx * dx;
            v[1] += dx * dx * dx;
        }
        const int b = off[x], d = outdeg[x];
        for (int j = sub; j < d; j += 8) {
            const unsigned long long dy = (unsigned)deg[adj[b + j]];
            v[2] += 2 * dx * dy;
            if (tri) {
                const unsigned long long t = tri[b + j];
                v[3] += t * (dx + dy);
                v[4] += 2 * t * t;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 5; j++) {
        const unsigned long long s = gpm_warp_sum(v[j]);
        if ((threadIdx.x & 31) == 0 && s) atomicAdd(&sum[j], s);
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int at[6] = {H_CHERRY, H_STAR3, H_PATH4, H_PAW, H_DIAMOND, 0};
        const bool time = threadIdx.x == 5;
        const unsigned long long x = time ? (gpm_globaltimer() - t0) * (blockDim.x / 32) : sum[threadIdx.x];
        if (x) atomicAdd(time ? busy : &hom[at[threadIdx.x]], x);
    }
}

struct Cycle4Params {
    const int32_t* __restrict__ indptr;
    const int32_t* __restrict__ indices;
    const int32_t* __restrict__ deg;
    const int32_t* __restrict__ outdeg;
    const int32_t* __restrict__ order;    // largest degree first
    int32_t n;
    unsigned int* counters;               // n per block (global variant), zero
    unsigned long long* ticket;
    unsigned long long* out;              // += 8 x cycles
    unsigned long long* busy;             // this launch's warp time
};

// one scan of the paths u - v - w with v, w before u; take: c(w) is read and
// zeroed, the first lane to reach w adding C(c(w), 2)
template <bool SMEM>
__device__ __forceinline__ void c4_scan(const Cycle4Params& p, unsigned int* cnt, int u, int du, bool take,
                                        unsigned long long& sum) {
    const int lane = threadIdx.x & 31;
    const int end = p.indptr[u + 1];
    for (int i = p.indptr[u] + (threadIdx.x >> 5); i < end; i += C4_THREADS / 32) {
        const int v = p.indices[i];
        const int dv = p.deg[v];
        if (dv > du || (dv == du && v > u)) continue;
        const int ve = p.indptr[v + 1];
        for (int q = p.indptr[v] + lane; q < ve; q += 32) {
            const int w = p.indices[q];
            const int dw = p.deg[w];
            if (dw > du || (dw == du && w >= u)) continue;
            if (!take) {
                if (SMEM) atomicAdd(&cnt[w >> 1], 1u << (16 * (w & 1)));
                else atomicAdd(&cnt[w], 1u);
            } else if (SMEM) {
                // (both counters of the word; a plain look spares the repeats)
                if (*(volatile unsigned int*)&cnt[w >> 1]) {
                    const unsigned int c = atomicExch(&cnt[w >> 1], 0u);
                    const unsigned long long lo = c & 0xffffu, hi = c >> 16;
                    sum += (lo * lo - lo + hi * hi - hi) / 2;
                }
            } else if (*(volatile unsigned int*)&cnt[w]) {
                const unsigned long long c = atomicExch(&cnt[w], 0u);
                if (c) sum += c * (c - 1) / 2;
            }
        }
    }
}

template <bool SMEM>
__global__ void __launch_bounds__(C4_THREADS) k_cycle4(Cycle4Params p) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_u[32];
    __shared__ unsigned s_mask;
    // (end minus start, added up modulo 2^64: nothing is held over the loops)
    if (threadIdx.x == 0) atomicAdd(p.busy, 0ull - gpm_globaltimer() * (C4_THREADS / 32));
    unsigned int* cnt = SMEM ? smem : p.counters + (size_t)blockIdx.x * p.n;
    if (SMEM)
        for (int i = threadIdx.x; i < (p.n + 1) / 2; i += C4_THREADS) cnt[i] = 0u;
    unsigned long long sum = 0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x < 32) {
            unsigned long long t = 0;
            if (threadIdx.x == 0) t = atomicAdd(p.ticket, 1ull);
            t = __shfl_sync(GPM_FULL_MASK, t, 0);
            const bool single = t < C4_SINGLE;
            const unsigned long long pos = single ? t : C4_SINGLE + (t - C4_SINGLE) * 32 + threadIdx.x;
            int u = -1;
            if (pos < (unsigned long long)p.n && (!single || threadIdx.x == 0)) {
                u = p.order[pos];
                // a cycle's last vertex has two neighbours before it
                if (p.deg[u] - p.outdeg[u] < 2) u = -1;
            }
            s_u[threadIdx.x] = u;
            const unsigned m = __ballot_sync(GPM_FULL_MASK, u >= 0);
            const bool past = (single ? t : C4_SINGLE + (t - C4_SINGLE) * 32) >= (unsigned long long)p.n;
            if (threadIdx.x == 0) s_mask = m;
            if (threadIdx.x == 0 && past) s_u[0] = -2;
        }
        __syncthreads();
        unsigned m = s_mask;
        if (s_u[0] == -2) break;
        for (; m; m &= m - 1u) {
            const int u = s_u[__ffs(m) - 1];
            const int du = p.deg[u];
            c4_scan<SMEM>(p, cnt, u, du, false, sum);
            __syncthreads();
            c4_scan<SMEM>(p, cnt, u, du, true, sum);
            __syncthreads();
        }
    }
    sum = gpm_warp_sum(sum);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(p.out, 8 * sum);
    if (threadIdx.x == 0) atomicAdd(p.busy, gpm_globaltimer() * (C4_THREADS / 32));
}

// ------------------------------------------------------------------- host

bool motif_sparse_applies(gpm_graph* g, int k) {
    if ((k != 3 && k != 4) || g->n < 1) return false;
    // every homomorphism count is at most (sum of degrees) x (largest degree)^(k-2)
    double bound = (double)g->nnz;
    for (int i = 2; i < k; i++) bound *= (double)std::max(g->max_deg, 1);
    if (bound >= 9.0e18 || g->max_deg >= 65536) return false;   // (16-bit counters)
    // (int32 offsets of the padded orientation)
    if (g->nnz / 2 + 3 * std::min<long long>(g->n, g->nnz / 2) >= INT32_MAX) return false;
    if (g->max_outdeg > 1024) return false;                     // no list path
    const bool built = g->dag_ready;
    ensure_dag(g);
    if (g->max_outdeg <= 1024) return true;
    if (!built) release_dag(g);                                 // the walk does not use it
    return false;
}

void run_motif_sparse(gpm_graph* g, int k, uint64_t* counts_out) {
    const HomTable& t = hom_table(k);
    cudaStream_t s = g->stream;
    struct Result {
        Control ctl;
        unsigned long long hom[HOM_N];
        unsigned long long ticket;
    };
    const int32_t* order = ensure_root_order(g, GPM_APP_MOTIF);
    ensure_root_order(g, GPM_APP_CLIQUE);
    const long long dag_entries = g->dag_adj.bytes / sizeof(int32_t);
    const bool smem = g->n <= C4_SMEM_N;
    // (counters in global memory: 8 GB at most, one block at least)
    const int blocks = smem ? g->num_sms
                            : (int)std::max<long long>(1, std::min<long long>(g->num_sms, (1ll << 31) / g->n));
    const size_t tri_bytes = (sizeof(unsigned int) * (size_t)dag_entries + 255) & ~size_t(255);
    const size_t cnt_bytes = k == 4 && !smem ? sizeof(unsigned int) * (size_t)g->n * blocks : 0;
    g->scratch_small.ensure(sizeof(Result));
    Result* r = g->scratch_small.as<Result>();
    unsigned int* tri = nullptr;
    GPM_CUDA(cudaMemsetAsync(r, 0, sizeof(Result), s));
    if (k == 4) {
        g->scratch_slab.ensure(tri_bytes + cnt_bytes);
        tri = g->scratch_slab.as<unsigned int>();
        GPM_CUDA(cudaMemsetAsync(tri, 0, tri_bytes + cnt_bytes, s));
    }
    Launches made;
    GPM_CUDA(cudaEventRecord(g->ev0, s));
    launch_clique_nonedge(g, 3, k, &r->ctl, made, tri);
    const int per_sm = g->cfg.blocks_per_sm > 0 ? std::min(g->cfg.blocks_per_sm, 8) : 8;
    const Grid sums{std::max(1, std::min((g->n + 31) / 32, g->num_sms * per_sm)), 8};
    k_edge_sums<<<sums.blocks, sums.warps_per_block * 32, 0, s>>>(
        g->dag_off.as<int32_t>(), g->dag_adj.as<int32_t>(), g->dag_outdeg.as<int32_t>(), g->degree.as<int32_t>(), tri,
        g->n, r->hom, made.add(&r->ctl, sums));
    GPM_CUDA(cudaGetLastError());
    if (k == 4) {
        Cycle4Params p{};
        p.indptr = g->indptr.as<int32_t>();
        p.indices = g->indices.as<int32_t>();
        p.deg = g->degree.as<int32_t>();
        p.outdeg = g->dag_outdeg.as<int32_t>();
        p.order = order;
        p.n = g->n;
        p.counters = tri + tri_bytes / sizeof(unsigned int);
        p.ticket = &r->ticket;
        p.out = &r->hom[H_CYCLE4];
        p.busy = made.add(&r->ctl, Grid{blocks, C4_THREADS / 32});
        if (smem) {
            const size_t bytes = sizeof(uint32_t) * (size_t)((g->n + 1) / 2);
            allow_shared((const void*)k_cycle4<true>, bytes);
            k_cycle4<true><<<blocks, C4_THREADS, bytes, s>>>(p);
        } else {
            k_cycle4<false><<<blocks, C4_THREADS, 0, s>>>(p);
        }
        GPM_CUDA(cudaGetLastError());
    }
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
    st.busy_warp_ns = made.busy_ns(h.ctl);
    st.kernel_launches = made.n;
    st.grid_blocks = made.grid[0].blocks;
    st.warps_per_block = made.grid[0].warps_per_block;
    g->stats = st;
    unsigned long long* hom = h.hom;
    const unsigned long long cherries = hom[H_CHERRY];
    hom[H_POINT] = (unsigned long long)g->n;
    hom[H_EDGE] = (unsigned long long)g->nnz;
    hom[H_TRI] = 6 * h.ctl.counts[3];
    hom[H_K4] = k == 4 ? 24 * h.ctl.counts[4] : 0;
    // closed walks of four steps that are no cycle: back and forth
    hom[H_CYCLE4] += 2 * cherries - (unsigned long long)g->nnz;
    hom_combine(t, hom, counts_out);
}

}  // namespace gpm
