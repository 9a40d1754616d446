// sched.cu -- the learned scheduler (hot-path row A10).
//
// Not part of the paper: a small MLP predicts each root's enumeration-subtree
// size from 8 per-root features; its predictions order the roots heaviest
// first and pre-split the heaviest ones into several work units before the
// enumeration starts, so that fewer splits are left to the in-kernel donation
// layer.  The network only changes which warp runs which part of the search,
// never what is counted.
//
//   features (FP32, per vertex v, for subgraph size k):
//     f0 log1p d(v)            f1 log1p d+(v) (degree-ordered out-degree)
//     f2 log1p |{u in N(v): u > v}|       (motif root's first extension set)
//     f3 log1p sum_{u in N(v)} d(u)       f4 log1p sum_{u in N(v), u > v} d(u)
//     f5 log1p triangles whose lowest (degree, id) vertex is v
//     f6 log1p core number of v           f7 k / 8 (one network serves several k)
//   network: 8 -> 64 -> 64 -> 1, ReLU, BF16 weights, FP32 activations and
//   accumulation; trained with MSE on log-sizes and Adam on FP32 master weights.
//
// The MLP is ~5k parameters and runs over at most a few hundred thousand
// roots (~0.3 GFLOP): microseconds against seconds of enumeration, so it is
// plain FP32 SIMT code with the weights broadcast from shared memory.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <string>
#include <vector>

#include "common.cuh"

namespace gpm {

constexpr int MLP_IN = 8, MLP_H = 64;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MLP_H * MLP_IN, OFF_W2 = OFF_B1 + MLP_H,
              OFF_B2 = OFF_W2 + MLP_H * MLP_H, OFF_W3 = OFF_B2 + MLP_H, OFF_B3 = OFF_W3 + MLP_H,
              MLP_NPARAM = OFF_B3 + 1;
static_assert(MLP_NPARAM == GPM_MLP_PARAMS, "parameter count");

// ------------------------------------------------------------- features

// triangles rooted at v in the degree orientation: sum over u in N+(v) of
// |N+(v) & N+(u)|.  Warp per v.  Up to TRI_LIST entries N+(v) lies in shared
// memory and eight lanes take a list N+(u) with 16-byte loads (the lists are
// padded and aligned for it); above, the whole warp takes a list, whose
// consecutive entries search nearly the same words of N+(v), in L1.
//
// Bound: the latency of the searches.  All root features, every list by whole
// warps / by eight lanes, in shared memory up to 1,024 / this: R-MAT 2^16 16.4 /
// 2.2 / 2.2 ms (the first with the core numbers of then), random graph of 30,000
// vertices and degree 1,000 61 / 57 / 38, K_1100 14.2 / 17.4 / 13.0, random graph
// of 8,192 vertices and degree 3,500 257 / 753 / 229.
constexpr int TRI_LIST = 256;
constexpr int TRI_THREADS = 256;
__global__ void __launch_bounds__(TRI_THREADS, 8) k_tri_root(const int32_t* __restrict__ off,
                                                             const int32_t* __restrict__ adj,
                                                             const int32_t* __restrict__ outdeg, int32_t n,
                                                             float* __restrict__ tri) {
    __shared__ int32_t s_list[TRI_THREADS / 32][TRI_LIST];
    const int lane = threadIdx.x & 31;
    int32_t* sl = s_list[threadIdx.x >> 5];
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long v = warp; v < n; v += nw) {
        const int b = off[v], d = outdeg[v];
        const bool small = d <= TRI_LIST;
        if (small)
            for (int t = lane; t < d; t += 32) sl[t] = adj[b + t];
        __syncwarp();
        long long c = 0;
        // the entries of N+(u) for all u in N+(v), searched in `list` = N+(v)
        auto found = [d](const auto* list, int x) {
            int lo = 0, hi = d - 1;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (list[mid] < x) lo = mid + 1; else hi = mid;
            }
            return list[lo] == x ? 1 : 0;
        };
        if (!small) {
            const int32_t* list = adj + b;
            for (int i = 0; i < d; i++) {
                const int u = list[i];
                const int ub = off[u], du = outdeg[u];
                for (int t = lane; t < du; t += 32) c += found(list, adj[ub + t]);
            }
        } else {
            for (int i = lane >> 3; i < d; i += 4) {
                const int u = sl[i];
                const int ub = off[u], du = outdeg[u];
                for (int t = 4 * (lane & 7); t < du; t += 32) {
                    const int4 x4 = *reinterpret_cast<const int4*>(adj + ub + t);   // padding is above every id
                    c += found(sl, x4.x) + found(sl, x4.y) + found(sl, x4.z) + found(sl, x4.w);
                }
            }
        }
        c = gpm_warp_sum(c);
        if (lane == 0) tri[v] = (float)c;
        __syncwarp();
    }
}

// Core numbers by peeling (the k-core decomposition), in one cooperative
// launch: at level c every remaining vertex whose remaining degree is <= c gets
// core number c and is removed, which lowers its remaining neighbours' degrees.
// The vertices that fall to c that way (each noticed by the decrement that
// takes it from c + 1 to c) form the next round of the level; when a round is
// empty, a scan of all vertices finds the next level, the smallest remaining
// degree, and its first round.  Rounds are separated by grid barriers.
//
// Bound: the barriers, about one per round and level.  Up to CORE_CLUSTER_N
// vertices the launch is one cluster of eight blocks, whose barrier is a
// hardware one; above, one block per SM (the scans of a level need the threads).
// Between two barriers a round is a chain of dependent loads, so each lane
// keeps four entries in flight and a short round spreads each list over up to a
// block (eight lanes per vertex left a hub's list serial), and the last level
// ends without its round: its vertices lower nothing.
// All root features: R-MAT 2^14 2.1 -> 0.87 ms, 2^16 4.9 -> 2.25, 10^6-vertex
// Chung-Lu 62 -> 15.9.  One launch per pass over all vertices, with the host
// reading a flag in between, took 9.4, 16.4 and 254 ms.
constexpr int CORE_THREADS = 512;
constexpr int CORE_CLUSTER = 8;
constexpr int CORE_CLUSTER_N = 1 << 17;

struct CoreState {
    int n_queue[3];      // sizes of the rounds: current, next, and the one being zeroed
    int min_left[2];     // smallest remaining degree found by a scan (two in turn)
};

template <bool CLUSTER>
__device__ __forceinline__ void core_sync() {
    if constexpr (CLUSTER) cooperative_groups::this_cluster().sync();
    else cooperative_groups::this_grid().sync();
}

template <bool CLUSTER>
__global__ void __launch_bounds__(CORE_THREADS) k_core(const int32_t* __restrict__ indptr,
                                                       const int32_t* __restrict__ indices, int32_t n,
                                                       int32_t* rem, int32_t* core, int32_t* queue0, int32_t* queue1,
                                                       CoreState* st) {
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    for (long long v = tid; v < n; v += nt) {
        rem[v] = indptr[v + 1] - indptr[v];
        core[v] = -1;
    }
    if (tid == 0) {
        st->n_queue[0] = st->n_queue[1] = st->n_queue[2] = 0;
        st->min_left[0] = st->min_left[1] = INT32_MAX;
    }
    core_sync<CLUSTER>();
    int c = 0, round = 0, scan = 0;
    for (;;) {
        // the vertices of level c, and the smallest degree above it
        int least = INT32_MAX;
        for (long long v0 = tid; v0 < n; v0 += 4 * nt) {
            int cs[4], rs[4];
#pragma unroll
            for (int z = 0; z < 4; z++) {
                const long long v = v0 + z * nt;
                cs[z] = v < n ? core[v] : 0;
                rs[z] = v < n ? rem[v] : 0;
            }
#pragma unroll
            for (int z = 0; z < 4; z++) {
                if (cs[z] >= 0) continue;
                const long long v = v0 + z * nt;
                if (rs[z] <= c) {
                    core[v] = c;
                    (round & 1 ? queue1 : queue0)[atomicAdd(&st->n_queue[round % 3], 1)] = (int32_t)v;
                } else {
                    least = min(least, rs[z]);
                }
            }
        }
        least = (int)__reduce_min_sync(GPM_FULL_MASK, (unsigned)least);
        if ((threadIdx.x & 31) == 0 && least != INT32_MAX) atomicMin(&st->min_left[scan & 1], least);
        core_sync<CLUSTER>();
        const int left = *(volatile int*)&st->min_left[scan & 1];
        const bool none = *(volatile int*)&st->n_queue[round % 3] == 0;
        if (tid == 0) st->min_left[(scan + 1) & 1] = INT32_MAX;
        scan++;
        if (left == INT32_MAX) break;    // every vertex that was left has level c: nothing to lower
        for (;;) {
            const int m = *(volatile int*)&st->n_queue[round % 3];
            if (!m) break;
            const int32_t* q = round & 1 ? queue1 : queue0;
            int32_t* next = round & 1 ? queue0 : queue1;
            // 2^sh lanes per removed vertex: at least eight, more while the round
            // leaves threads over, at most a block (a divisor of the thread count)
            int sh = 3;
            while ((2 << sh) <= CORE_THREADS && ((long long)m << (sh + 1)) <= nt) sh++;
            const int w = 1 << sh;
            for (long long i = tid >> sh; i < m; i += nt >> sh) {
                const int v = __ldcg(q + i);
                const long long e = indptr[v + 1];
                for (long long t = indptr[v] + (tid & (w - 1)); t < e; t += 4 * w) {
                    int us[4], old[4];
#pragma unroll
                    for (int z = 0; z < 4; z++) us[z] = t + z * w < e ? indices[t + z * w] : -1;
#pragma unroll
                    for (int z = 0; z < 4; z++) old[z] = us[z] < 0 ? 0 : *(volatile int*)&core[us[z]];
#pragma unroll
                    for (int z = 0; z < 4; z++) old[z] = old[z] < 0 ? atomicSub(&rem[us[z]], 1) : -1;
#pragma unroll
                    for (int z = 0; z < 4; z++)
                        if (old[z] == c + 1) {
                            *(volatile int*)&core[us[z]] = c;
                            next[atomicAdd(&st->n_queue[(round + 1) % 3], 1)] = us[z];
                        }
                }
            }
            if (tid == 0) st->n_queue[(round + 2) % 3] = 0;
            core_sync<CLUSTER>();
            round++;
        }
        // (the rounds of level c can have brought vertices down to c + 1)
        c = none ? left : c + 1;
        core_sync<CLUSTER>();
    }
}

__global__ void k_features(const int32_t* __restrict__ indptr, const int32_t* __restrict__ indices,
                           const int32_t* __restrict__ deg, const int32_t* __restrict__ outdeg,
                           const float* __restrict__ tri, const int32_t* __restrict__ core, int32_t n, int k,
                           float* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long v = warp; v < n; v += nw) {
        const int b = indptr[v], e = indptr[v + 1];
        double s_all = 0, s_up = 0;
        int c_up = 0;
        // four entries per lane in flight: a hub's list is the kernel's time
        for (int t = b + lane; t < e; t += 128) {
            int us[4], ds[4];
#pragma unroll
            for (int z = 0; z < 4; z++) us[z] = t + 32 * z < e ? indices[t + 32 * z] : -1;
#pragma unroll
            for (int z = 0; z < 4; z++) ds[z] = us[z] >= 0 ? deg[us[z]] : 0;
#pragma unroll
            for (int z = 0; z < 4; z++) {
                s_all += ds[z];
                if (us[z] > v) {
                    s_up += ds[z];
                    c_up++;
                }
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            s_all += __shfl_xor_sync(GPM_FULL_MASK, s_all, o);
            s_up += __shfl_xor_sync(GPM_FULL_MASK, s_up, o);
            c_up += __shfl_xor_sync(GPM_FULL_MASK, c_up, o);
        }
        if (lane == 0) {
            float* f = out + v * MLP_IN;
            f[0] = log1pf((float)(e - b));
            f[1] = log1pf((float)outdeg[v]);
            f[2] = log1pf((float)c_up);
            f[3] = (float)log1p(s_all);
            f[4] = (float)log1p(s_up);
            f[5] = log1pf(tri[v]);
            f[6] = log1pf((float)core[v]);
            f[7] = (float)k / 8.f;
        }
    }
}

static int blocks_for(int64_t items_x32, int threads, int sms) {
    int64_t b = (items_x32 + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)sms * 32));
}

// core numbers of every vertex into d_core
static void core_numbers(gpm_graph* g, int32_t* d_core, DevBuf& tmp) {
    int32_t n = g->n;
    tmp.ensure(sizeof(int32_t) * 3 * (size_t)n + sizeof(CoreState));
    int32_t* rem = tmp.as<int32_t>();
    int32_t *q0 = rem + n, *q1 = q0 + n;
    CoreState* st = reinterpret_cast<CoreState*>(q1 + n);
    const int32_t *indptr = g->indptr.as<int32_t>(), *indices = g->indices.as<int32_t>();
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.blockDim = dim3(CORE_THREADS);
    cfg.stream = g->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (n <= CORE_CLUSTER_N) {
        cfg.gridDim = dim3(CORE_CLUSTER);
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim = {CORE_CLUSTER, 1, 1};
        GPM_CUDA(cudaLaunchKernelEx(&cfg, k_core<true>, indptr, indices, n, rem, d_core, q0, q1, st));
    } else {
        cfg.gridDim = dim3(g->num_sms);
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        GPM_CUDA(cudaLaunchKernelEx(&cfg, k_core<false>, indptr, indices, n, rem, d_core, q0, q1, st));
    }
}

void root_features(gpm_graph* g, int k, float* d_out) {
    ensure_dag(g);
    cudaStream_t s = g->stream;
    DevBuf tri, core, tmp;
    tri.ensure(sizeof(float) * std::max(g->n, 1));
    core.ensure(sizeof(int32_t) * std::max(g->n, 1));
    if (g->n > 0) {
        core_numbers(g, core.as<int32_t>(), tmp);
        k_tri_root<<<blocks_for((int64_t)g->n * 32, TRI_THREADS, g->num_sms), TRI_THREADS, 0, s>>>(
            g->dag_off.as<int32_t>(), g->dag_adj.as<int32_t>(), g->dag_outdeg.as<int32_t>(), g->n, tri.as<float>());
        k_features<<<blocks_for((int64_t)g->n * 32, 256, g->num_sms), 256, 0, s>>>(
            g->indptr.as<int32_t>(), g->indices.as<int32_t>(), g->degree.as<int32_t>(), g->dag_outdeg.as<int32_t>(),
            tri.as<float>(), core.as<int32_t>(), g->n, k, d_out);
        GPM_CUDA(cudaGetLastError());
    }
    GPM_CUDA(cudaStreamSynchronize(s));
}

// ------------------------------------------------------------------ MLP

__device__ __forceinline__ void load_weights(const uint16_t* __restrict__ w, float* W) {
    for (int i = threadIdx.x; i < MLP_NPARAM; i += blockDim.x) {
        __nv_bfloat16_raw r;
        r.x = w[i];
        W[i] = __bfloat162float(__nv_bfloat16(r));
    }
    __syncthreads();
}

// thread per sample; y = w3 . relu(W2 relu(W1 x + b1) + b2) + b3
__global__ void __launch_bounds__(256) k_mlp_forward(const uint16_t* __restrict__ w, const float* __restrict__ x,
                                                     long long n, float* __restrict__ y) {
    __shared__ float W[MLP_NPARAM];
    load_weights(w, W);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        float xi[MLP_IN];
#pragma unroll
        for (int q = 0; q < MLP_IN; q++) xi[q] = x[i * MLP_IN + q];
        float h1[MLP_H];
#pragma unroll
        for (int j = 0; j < MLP_H; j++) {
            float s = W[OFF_B1 + j];
#pragma unroll
            for (int q = 0; q < MLP_IN; q++) s = fmaf(W[OFF_W1 + j * MLP_IN + q], xi[q], s);
            h1[j] = fmaxf(s, 0.f);
        }
        float out = W[OFF_B3];
        for (int j = 0; j < MLP_H; j++) {
            float s = W[OFF_B2 + j];
#pragma unroll
            for (int q = 0; q < MLP_H; q++) s = fmaf(W[OFF_W2 + j * MLP_H + q], h1[q], s);
            out = fmaf(W[OFF_W3 + j], fmaxf(s, 0.f), out);
        }
        y[i] = out;
    }
}

// Gradients of mean_i (y_i - t_i)^2 over a minibatch of n samples.  A block of
// 256 threads takes BW_TILE samples at a time; every product of the pass is a
// small matrix product over shared memory with a register tile per thread:
//
//   z1 = x W1' + b1, z2 = relu(z1) W2' + b2, D1 = (D2 W2) .* [z1 > 0]   tile x 64, 4 x 2 per thread
//   dW2 += D2' relu(z1)   64 x 64, 4 x 4 per thread, kept over the block's tiles
//   dW1 += D1' x          64 x 8, 2 per thread
//
// and the block adds its sums to grad once (FP32 atomics).  grad and loss must
// be zero on entry.  Bound: the latency of the phases of one tile (a minibatch
// of 4,096 is one tile per block) and the atomics.  With one thread per sample
// and rows of dW2 per thread, 64 threads per block, it took 65 us at n = 4,096.
constexpr int BW_TILE = 32;
constexpr int BW_THREADS = 256;
constexpr int BW_S = MLP_H + 1;                      // row stride of the 64-wide arrays
constexpr int BW_SMEM = MLP_NPARAM + 3 + BW_TILE * MLP_IN + 4 * BW_TILE * BW_S + BW_TILE;
__global__ void __launch_bounds__(BW_THREADS) k_mlp_backward(const uint16_t* __restrict__ w,
                                                             const float* __restrict__ x, const float* __restrict__ t,
                                                             long long n, float* __restrict__ grad,
                                                             float* __restrict__ loss) {
    extern __shared__ float sh[];
    float* W = sh;                                   // MLP_NPARAM
    float* X = W + MLP_NPARAM + 3;                   // BW_TILE x 8
    float* H1 = X + BW_TILE * MLP_IN;                // relu(z1)
    float* H2 = H1 + BW_TILE * BW_S;                 // relu(z2)
    float* D2 = H2 + BW_TILE * BW_S;                 // dL/dz2
    float* D1 = D2 + BW_TILE * BW_S;                 // dL/dz1
    float* DY = D1 + BW_TILE * BW_S;                 // dL/dy
    load_weights(w, W);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float inv_n = 1.0f / (float)n;
    // tile x 64 products: samples s0 .. s0 + 3, neurons j0 and j0 + 32
    const int s0 = 4 * wid, j0 = lane;
    // 64 x 64 gradient: rows r0 .. r0 + 3, columns q0, q0 + 16, q0 + 32, q0 + 48
    const int r0 = 4 * (tid >> 4), q0 = tid & 15;
    float gW2[4][4], gW1[2] = {0.f, 0.f}, gb1 = 0.f, gb2 = 0.f, gw3 = 0.f, gb3 = 0.f, lsum = 0.f;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int q = 0; q < 4; q++) gW2[i][q] = 0.f;

    for (long long base = (long long)blockIdx.x * BW_TILE; base < n; base += (long long)gridDim.x * BW_TILE) {
        for (int i = tid; i < BW_TILE * MLP_IN; i += BW_THREADS)
            X[i] = base + i / MLP_IN < n ? x[base * MLP_IN + i] : 0.f;
        __syncthreads();
        // z1
#pragma unroll
        for (int jj = 0; jj < 2; jj++) {
            const int j = j0 + 32 * jj;
            float wj[MLP_IN];
#pragma unroll
            for (int q = 0; q < MLP_IN; q++) wj[q] = W[OFF_W1 + j * MLP_IN + q];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                float s = W[OFF_B1 + j];
#pragma unroll
                for (int q = 0; q < MLP_IN; q++) s = fmaf(wj[q], X[(s0 + i) * MLP_IN + q], s);
                H1[(s0 + i) * BW_S + j] = fmaxf(s, 0.f);
            }
        }
        __syncwarp();                                // (a warp's samples are its own until D1 is there)
        // z2
        float z[4][2];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            z[i][0] = W[OFF_B2 + j0];
            z[i][1] = W[OFF_B2 + j0 + 32];
        }
#pragma unroll 8
        for (int q = 0; q < MLP_H; q++) {
            const float w0 = W[OFF_W2 + j0 * MLP_H + ((q + j0) & 63)], w1 = W[OFF_W2 + (j0 + 32) * MLP_H + ((q + j0) & 63)];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float h = H1[(s0 + i) * BW_S + ((q + j0) & 63)];
                z[i][0] = fmaf(w0, h, z[i][0]);
                z[i][1] = fmaf(w1, h, z[i][1]);
            }
        }
        // y, dy, D2
        const float v0 = W[OFF_W3 + j0], v1 = W[OFF_W3 + j0 + 32];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const float h0 = fmaxf(z[i][0], 0.f), h1 = fmaxf(z[i][1], 0.f);
            const float y = gpm_warp_sum(fmaf(v0, h0, v1 * h1)) + W[OFF_B3];
            const long long g = base + s0 + i;
            const float diff = g < n ? y - t[g] : 0.f;
            const float dy = 2.f * diff * inv_n;
            if (lane == 0) {
                DY[s0 + i] = dy;
                lsum += diff * diff;
            }
            H2[(s0 + i) * BW_S + j0] = h0;
            H2[(s0 + i) * BW_S + j0 + 32] = h1;
            D2[(s0 + i) * BW_S + j0] = z[i][0] > 0.f ? dy * v0 : 0.f;
            D2[(s0 + i) * BW_S + j0 + 32] = z[i][1] > 0.f ? dy * v1 : 0.f;
        }
        __syncwarp();
        // D1
        float d[4][2];
#pragma unroll
        for (int i = 0; i < 4; i++) d[i][0] = d[i][1] = 0.f;
#pragma unroll 8
        for (int q = 0; q < MLP_H; q++) {
            const float w0 = W[OFF_W2 + q * MLP_H + j0], w1 = W[OFF_W2 + q * MLP_H + j0 + 32];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float e = D2[(s0 + i) * BW_S + q];
                d[i][0] = fmaf(e, w0, d[i][0]);
                d[i][1] = fmaf(e, w1, d[i][1]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            D1[(s0 + i) * BW_S + j0] = H1[(s0 + i) * BW_S + j0] > 0.f ? d[i][0] : 0.f;
            D1[(s0 + i) * BW_S + j0 + 32] = H1[(s0 + i) * BW_S + j0 + 32] > 0.f ? d[i][1] : 0.f;
        }
        __syncthreads();
        // dW2
#pragma unroll 4
        for (int s = 0; s < BW_TILE; s++) {
            float e[4], h[4];
#pragma unroll
            for (int i = 0; i < 4; i++) e[i] = D2[s * BW_S + r0 + i];
#pragma unroll
            for (int q = 0; q < 4; q++) h[q] = H1[s * BW_S + q0 + 16 * q];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int q = 0; q < 4; q++) gW2[i][q] = fmaf(e[i], h[q], gW2[i][q]);
        }
        // dW1: entries tid and tid + 256 (row j, column q); the vectors: a warp pair each
        {
            const int j = tid >> 3, q = tid & 7;
#pragma unroll 8
            for (int s = 0; s < BW_TILE; s++) {
                const float xv = X[s * MLP_IN + q];
                gW1[0] = fmaf(D1[s * BW_S + j], xv, gW1[0]);
                gW1[1] = fmaf(D1[s * BW_S + j + 32], xv, gW1[1]);
            }
        }
        const int j = tid & 63, part = tid >> 6;     // 0: b1, 1: b2, 2: w3, 3: b3
        if (part == 0) {
            for (int s = 0; s < BW_TILE; s++) gb1 += D1[s * BW_S + j];
        } else if (part == 1) {
            for (int s = 0; s < BW_TILE; s++) gb2 += D2[s * BW_S + j];
        } else if (part == 2) {
            for (int s = 0; s < BW_TILE; s++) gw3 = fmaf(DY[s], H2[s * BW_S + j], gw3);
        } else if (j == 0) {
            for (int s = 0; s < BW_TILE; s++) gb3 += DY[s];
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int q = 0; q < 4; q++) atomicAdd(&grad[OFF_W2 + (r0 + i) * MLP_H + q0 + 16 * q], gW2[i][q]);
    atomicAdd(&grad[OFF_W1 + tid], gW1[0]);
    atomicAdd(&grad[OFF_W1 + tid + 256], gW1[1]);
    const int j = tid & 63, part = tid >> 6;
    if (part == 0) atomicAdd(&grad[OFF_B1 + j], gb1);
    else if (part == 1) atomicAdd(&grad[OFF_B2 + j], gb2);
    else if (part == 2) atomicAdd(&grad[OFF_W3 + j], gw3);
    else if (j == 0) atomicAdd(&grad[OFF_B3], gb3);
    if (lane == 0) atomicAdd(loss, lsum * inv_n);
}

// Adam (Kingma & Ba 2015), bias-corrected; master weights FP32, BF16 copy out
__global__ void k_mlp_adam(float* __restrict__ master, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ grad, int step, float lr, float beta1, float beta2, float eps,
                           uint16_t* __restrict__ w) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MLP_NPARAM) return;
    const float g = grad[i];
    const float mi = beta1 * m[i] + (1.f - beta1) * g;
    const float vi = beta2 * v[i] + (1.f - beta2) * g * g;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / (1.f - powf(beta1, (float)step));
    const float vh = vi / (1.f - powf(beta2, (float)step));
    const float p = master[i] - lr * mh / (sqrtf(vh) + eps);
    master[i] = p;
    __nv_bfloat16 b = __float2bfloat16_rn(p);
    w[i] = __nv_bfloat16_raw(b).x;
}

void mlp_forward(const uint16_t* w, const float* x, int64_t n, float* y, cudaStream_t s) {
    if (n <= 0) return;
    int dev = 0, sms = 0;
    GPM_CUDA(cudaGetDevice(&dev));
    GPM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8);
    k_mlp_forward<<<blocks, 256, 0, s>>>(w, x, n, y);
    GPM_CUDA(cudaGetLastError());
}

void mlp_grad(const uint16_t* w, const float* x, const float* t, int64_t n, float* grad, float* loss, cudaStream_t s) {
    GPM_CUDA(cudaMemsetAsync(grad, 0, sizeof(float) * MLP_NPARAM, s));
    GPM_CUDA(cudaMemsetAsync(loss, 0, sizeof(float), s));
    if (n <= 0) return;
    int dev = 0, sms = 0;
    GPM_CUDA(cudaGetDevice(&dev));
    GPM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = sizeof(float) * BW_SMEM;
    allow_shared((const void*)k_mlp_backward, smem);
    const int blocks = (int)std::min<int64_t>((n + BW_TILE - 1) / BW_TILE, (int64_t)sms * 2);
    k_mlp_backward<<<blocks, BW_THREADS, smem, s>>>(w, x, t, n, grad, loss);
    GPM_CUDA(cudaGetLastError());
}

void mlp_adam(float* master, float* m, float* v, const float* grad, int step, float lr, uint16_t* w, cudaStream_t s) {
    k_mlp_adam<<<(MLP_NPARAM + 255) / 256, 256, 0, s>>>(master, m, v, grad, step, lr, 0.9f, 0.999f, 1e-8f, w);
    GPM_CUDA(cudaGetLastError());
}

// ------------------------------------------------------------ schedule

// monotone 16-bit key of a float score, descending order -> ascending key
__device__ __forceinline__ uint32_t score_key(float f) {
    uint32_t u = __float_as_uint(f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);   // order-preserving map to uint32
    return 0xffffu - (u >> 16);
}

__global__ void k_score_hist(const float* __restrict__ score, const int32_t* __restrict__ roots, long long n,
                             int32_t* __restrict__ hist) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        atomicAdd(&hist[score_key(score[roots ? roots[i] : i])], 1);
}

__global__ void k_score_scatter(const float* __restrict__ score, const int32_t* __restrict__ roots, long long n,
                                int32_t* __restrict__ cursor, int32_t* __restrict__ order) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int v = roots ? roots[i] : (int)i;
        order[atomicAdd(&cursor[score_key(score[v])], 1)] = v;
    }
}

// roots (or all vertices) ordered by score descending (bucketed by the top 16
// bits of the float; ties in no particular order)
void order_by_score(gpm_graph* g, const float* d_score, const int32_t* d_roots, int64_t n_roots, DevBuf& out) {
    cudaStream_t s = g->stream;
    out.ensure(sizeof(int32_t) * std::max<int64_t>(n_roots, 1));
    DevBuf hist, cur, tmp;
    hist.ensure(sizeof(int32_t) * 65537);
    cur.ensure(sizeof(int32_t) * 65537);
    GPM_CUDA(cudaMemsetAsync(hist.ptr, 0, sizeof(int32_t) * 65537, s));
    if (n_roots > 0) {
        const int blocks = std::max(1, (int)std::min<int64_t>((n_roots + 255) / 256, (int64_t)g->num_sms * 16));
        k_score_hist<<<blocks, 256, 0, s>>>(d_score, d_roots, n_roots, hist.as<int32_t>());
        int64_t total = 0;
        exclusive_scan_i32(hist.as<int32_t>(), cur.as<int32_t>(), 65536, &total, s, tmp);
        k_score_scatter<<<blocks, 256, 0, s>>>(d_score, d_roots, n_roots, cur.as<int32_t>(), out.as<int32_t>());
        GPM_CUDA(cudaGetLastError());
    }
    GPM_CUDA(cudaStreamSynchronize(s));
}

}  // namespace gpm
