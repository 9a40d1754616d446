// clique_nonedge.cuh -- the cliques inside a candidate set, counted through
// its non-edges (device code of clique_nonedge.cu).
//
// A candidate set S of a traversal of size h (the vertices after it in the
// orientation, adjacent to all of it) holds, for every size j, i_j(S) sets of
// j pairwise adjacent members: the (h+j)-cliques below the traversal.  With H
// the complement graph on S (the non-edges) these are the independent sets of
// H, and for v in S
//
//     cliques in S  =  cliques in S without v  +  cliques in S that hold v,
//
// the latter being v together with the cliques of S \ H(v) \ {v}.  Taking for
// v the member with the most non-edges, what is left soon has none, or only
// pairwise disjoint ones, and then has a closed form:
//
//   * n members, b disjoint non-edges: i_j = sum_t 2^t C(b,t) C(n-2b, j-t);
//   * three sizes to go: i_2 = C(n,2) - e and
//     i_3 = C(n,3) - e (n-2) + w - t, with e_u the non-edges of member u, e
//     their sum / 2, w = sum_u C(e_u,2) and t the triangles of H;
//   * four sizes to go, by inclusion-exclusion over the sets of non-edges on at
//     most four members,
//     i_4 = C(n,4) - e C(n-2,2) + w (n-3) + (C(e,2) - w) - t (n-3)
//           - stars - paths + cycles + paws - diamonds + cliques   (4 vertices of H)
//     which all follow from the e_u and from the common non-neighbours of
//     pairs of members with two non-edges or more.
//
// Where more pairs are non-adjacent than adjacent, i_2 .. i_4 are counted
// directly as edges, triangles and 4-cliques among the members instead.
//
// A member without non-edges is in every closed form as a mere count, so a
// set is first reduced to its members that have one (the others' number is
// `a`), re-indexed 0 .. m-1.  The rows of H then have ceil(m/32) words and
// live in registers: lane t holds the rows of members t, t + 32, ...; a set
// is a warp-uniform bitmap, and e_u is one AND + POPC per word.
#pragma once

#include "common.cuh"

namespace gpm {

constexpr int NE_W = 4;              // most words of a re-indexed set: 128 members
constexpr int NE_BINOM_N = 1024;     // binomial table: n <= 1024, k <= 16
constexpr int NE_BINOM_K = GPM_CLIQUE_MAX_K + 1;
constexpr int NE_LEVELS = GPM_CLIQUE_MAX_K + 1;
// Four sizes to go: members with more non-edges than this are taken out first.
// Chung-Lu n = 10^6, k = 4..7, this launch alone: 1: 42.2 ms, 3: 41.3, 8: 36.4,
// 16: 34.4; R-MAT scale 16, k = 3..7: 7.1 / 6.8 / 5.7 / 5.7 ms.
constexpr int NE_SPARSE = 16;

// What one warp has counted.  The closed forms of three and four sizes to go
// are summed lane by lane without a reduction, as 24 times the cliques of
// size k_hi - q in acc[q] (24 makes every lane's share a whole number; a
// lane's sum may be negative, the warp's is not).  A set adds less than 2^41
// to acc[0] (members^4), less to the others; all are folded into `size` (with
// carry checks) at the end of a root (heavy launch) or of the warp (light
// launch: 32 members at most).  Where a root can have any number of sets --
// four sizes to go, or below a wide set -- ne_settle folds after a set that
// brought acc[0] or acc[1] past 2^57, so that none can wrap.
struct NeCount {
    unsigned long long size = 0;     // lane s: cliques of size s
    long long acc[5] = {0, 0, 0, 0, 0};
    unsigned long long wops = 0;     // candidate-word operations (lane 0's copy counts)
    int ovf = 0;
};

struct NeParams {
    int k_lo, k_hi;
    const unsigned long long* binom;   // [n][k], ~0ull where C(n, k) does not fit
};

__device__ __forceinline__ unsigned long long ne_mul(unsigned long long x, unsigned long long y, int& ovf) {
    if (__umul64hi(x, y)) ovf = 1;
    return x * y;
}

// n members, b of their pairs non-adjacent and these pairwise disjoint: lane
// s adds the cliques of size s = h + j, every j.
__device__ __forceinline__ void ne_matching(const NeParams& p, NeCount& c, int h, int n, int b, int lane) {
    const int j = lane - h;
    if (j < 0 || lane < p.k_lo || lane > p.k_hi) return;
    const unsigned long long* row = p.binom + (n - 2 * b) * NE_BINOM_K;
    unsigned long long sum = 0;
    int ovf = 0;
#pragma unroll 1
    for (int t = 0; t <= min(b, j); t++) {
        const unsigned long long x = row[j - t];
        if (t == 0) {
            sum = x;
            if (x == ~0ull) ovf = 1;
        } else if (x) {
            const unsigned long long y = p.binom[b * NE_BINOM_K + t];
            if (x == ~0ull || y == ~0ull) ovf = 1;
            sum = gpm_add_cc(sum, ne_mul(ne_mul(y, 1ull << t, ovf), x, ovf), ovf);
        }
    }
    c.size = gpm_add_cc(c.size, sum, ovf);
    c.ovf |= ovf;
}

// i_2, n and 1 of a set with two sizes to go (e2 = twice its non-edges)
__device__ __forceinline__ void ne_pairs(const NeParams& p, NeCount& c, unsigned n, unsigned e2, int lane) {
    const unsigned v = lane == p.k_hi ? (n * (n - 1) - e2) / 2 : lane == p.k_hi - 1 ? n : lane == p.k_hi - 2 ? 1u : 0u;
    c.size = gpm_add_cc(c.size, v, c.ovf);
}

// Fold the deferred sums into the sizes (all lanes must call).
__device__ __forceinline__ void ne_fold(const NeParams& p, NeCount& c, int lane) {
    unsigned long long v = 0;
#pragma unroll
    for (int q = 0; q < 5; q++) {
        const unsigned long long x = (unsigned long long)gpm_warp_sum(c.acc[q]);
        if (lane == p.k_hi - q) v = x / 24;
        c.acc[q] = 0;
    }
    c.size = gpm_add_cc(c.size, v, c.ovf);
}

// The same once a sum has passed 2^57, between two sets (all lanes must call).
__device__ __forceinline__ void ne_settle(const NeParams& p, NeCount& c, int lane) {
    const bool full = ((unsigned long long)(c.acc[0] + (1ll << 57)) | (unsigned long long)(c.acc[1] + (1ll << 57))) >> 58;
    if (__any_sync(GPM_FULL_MASK, full)) ne_fold(p, c, lane);
}

// The non-edges of the lane's members of S (members 32 x + lane).
template <int W>
__device__ __forceinline__ void ne_degrees(const uint32_t (&S)[W], const uint32_t (&h)[W][W], int (&e)[W], int lane) {
#pragma unroll
    for (int x = 0; x < W; x++) {
        int d = 0;
#pragma unroll
        for (int z = 0; z < W; z++) d += __popc(S[z] & h[x][z]);
        e[x] = (S[x] >> lane) & 1u ? d : 0;
    }
}

// The lane's member 32 x + lane: bits above it in word z
__device__ __forceinline__ uint32_t ne_above(int x, int z, int lane) {
    return z < x ? 0u : z > x ? 0xffffffffu : 0xfffffffeu << lane;
}

// Three sizes to go: all s members of a re-indexed set (rows h, Hs) and `a`
// members adjacent to all.  The triangles of H come from the lanes' upper
// rows, one loop step per non-edge; when more pairs are non-adjacent than
// adjacent (never asked with COMP) the triangles of the graph itself are
// counted the same way.
template <int W, bool COMP>
__device__ __forceinline__ void ne_triples(const NeParams& p, NeCount& c, const uint32_t (&S)[W], int s, int a,
                                           const uint32_t (&h)[W][W], const uint32_t* Hs, int lane) {
    int e[W];
    ne_degrees<W>(S, h, e, lane);
    int se = 0, see = 0;
#pragma unroll
    for (int x = 0; x < W; x++) {
        se += e[x];
        see += e[x] * (e[x] - 1);
    }
    // (warp-uniform)
    const bool comp = COMP || 2 * __reduce_add_sync(GPM_FULL_MASK, (unsigned)se) <= (unsigned)(s * (s - 1));
    const uint32_t flip = comp ? 0u : 0xffffffffu;
    int t = 0;
#pragma unroll
    for (int x = 0; x < W; x++) {
        if (!((S[x] >> lane) & 1u)) continue;
        uint32_t y[W];
        int up = 0;
#pragma unroll
        for (int z = 0; z < W; z++) {
            y[z] = S[z] & (h[x][z] ^ flip) & ne_above(x, z, lane);
            up += __popc(y[z]);
        }
        // the last of the upper neighbours closes no triangle above itself
#pragma unroll
        for (int z = x; z < W; z++) {
#pragma unroll 1
            while (y[z] && up > 1) {
                const uint32_t* r = Hs + (32 * z + __ffs(y[z]) - 1) * W;
                y[z] &= y[z] - 1u;
                up--;
#pragma unroll
                for (int q = z; q < W; q++) t += __popc(y[q] & (r[q] ^ flip));
            }
        }
    }
    const long long n = s + a;
    long long v = comp ? 12ll * (see - (long long)se * (n - 2)) - 24 * t : 24ll * t - 12ll * a * se;
    if (lane == 0) v += 4 * (n * (n - 1) * (n - 2) - (comp ? 0ll : (long long)s * (s - 1) * (s - 2)));
    c.acc[0] += v;
    c.acc[1] += (lane == 0 ? 12 * n * (n - 1) : 0ll) - 12 * se;
    if (lane == 0) {
        c.acc[2] += 24 * n;
        c.acc[3] += 24;
    }
    c.wops += (unsigned)(s * W);
}

// Four sizes to go: the set S (s members, e their non-edges, `all` their sum)
// and `a` members adjacent to all, by inclusion-exclusion.
template <int W>
__device__ __forceinline__ void ne_quads(const NeParams& p, NeCount& c, const uint32_t (&S)[W], int s, int a,
                                         const int (&e)[W], const uint32_t (&h)[W][W], const uint32_t* Hs, int lane) {
    int se = 0;
#pragma unroll
    for (int x = 0; x < W; x++) se += e[x];
    const long long all = (long long)__reduce_add_sync(GPM_FULL_MASK, (unsigned)se);
    const long long n = s + a;
    long long v4 = 0, v3 = 0;
    uint32_t two[W];
    int tt[W], pp[W];
#pragma unroll
    for (int x = 0; x < W; x++) {
        two[x] = __ballot_sync(GPM_FULL_MASK, e[x] >= 2);
        tt[x] = pp[x] = 0;
    }
    int c4 = 0, dd = 0, kk = 0;
    // pairs (u, v) of members with two non-edges or more: v uniform
#pragma unroll
    for (int zv = 0; zv < W; zv++) {
#pragma unroll 1
        for (uint32_t left = two[zv]; left; left &= left - 1u) {
            const int vb = __ffs(left) - 1;
            const uint32_t* r = Hs + (32 * zv + vb) * W;
            uint32_t hv[W];
#pragma unroll
            for (int z = 0; z < W; z++) hv[z] = r[z] & S[z];
            const int ev = __shfl_sync(GPM_FULL_MASK, e[zv], vb);
#pragma unroll
            for (int x = 0; x < W; x++) {
                uint32_t cw[W];
                int cod = 0;
#pragma unroll
                for (int z = 0; z < W; z++) {
                    cw[z] = h[x][z] & hv[z];
                    cod += __popc(cw[z]);
                }
                const bool self = x == zv && lane == vb;
                if (!((two[x] >> lane) & 1u) || self) cod = 0;
                const int cc = cod * (cod - 1) / 2;
                c4 += cc;
                if (((two[x] & hv[x]) >> lane) & 1u) {     // u, v not adjacent
                    pp[x] += ev - 1;
                    tt[x] += cod;
                    dd += cc;
                    if (cod >= 2) {                        // 4-cliques of H on u, v
#pragma unroll
                        for (int z = 0; z < W; z++) {
#pragma unroll 1
                            for (uint32_t y = cw[z]; y; y &= y - 1u) {
                                const uint32_t* ry = Hs + (32 * z + __ffs(y) - 1) * W;
#pragma unroll
                                for (int q = 0; q < W; q++) kk += __popc(cw[q] & ry[q]);
                            }
                        }
                    }
                }
            }
        }
    }
#pragma unroll
    for (int x = 0; x < W; x++) {
        const long long ex = e[x], t = tt[x];
        v4 += -4 * ex * (ex - 1) * (ex - 2) - 12 * (ex - 1) * (long long)pp[x] + 12 * t + 12 * t * (ex - 2) -
              4 * t * (n - 3) + 12 * (n - 4) * ex * (ex - 1) - 6 * ex * (n - 2) * (n - 3);
        v3 += 12 * (ex * (ex - 1) - ex * (n - 2)) - 4 * t;
    }
    v4 += 6ll * c4 - 12ll * dd + kk;
    if (lane == 0) {
        const long long m = all / 2;
        v4 += n * (n - 1) * (n - 2) * (n - 3) + 12 * m * (m - 1);
        v3 += 4 * n * (n - 1) * (n - 2);
    }
    c.acc[0] += v4;
    c.acc[1] += v3;
    c.acc[2] += (lane == 0 ? 12 * n * (n - 1) : 0ll) - 12 * se;
    if (lane == 0) {
        c.acc[3] += 24 * n;
        c.acc[4] += 24;
    }
    c.wops += (unsigned)(s * W);
}

// The same from the edges, triangles and 4-cliques of the graph (at their
// lowest member): where most pairs are non-adjacent.
template <int W>
__device__ __forceinline__ void ne_quads_graph(const NeParams& p, NeCount& c, const uint32_t (&S)[W], int s, int a,
                                               const int (&e)[W], const uint32_t (&h)[W][W], const uint32_t* Hs,
                                               int lane) {
    int se = 0;
#pragma unroll
    for (int x = 0; x < W; x++) se += e[x];
    const long long n = s + a, b = a;
    long long t = 0, q4 = 0;
#pragma unroll
    for (int x = 0; x < W; x++) {
        if (!((S[x] >> lane) & 1u)) continue;
        uint32_t y[W];
#pragma unroll
        for (int z = 0; z < W; z++) y[z] = S[z] & ~h[x][z] & ne_above(x, z, lane);
#pragma unroll
        for (int z = x; z < W; z++) {
#pragma unroll 1
            while (y[z]) {
                const uint32_t* r = Hs + (32 * z + __ffs(y[z]) - 1) * W;
                y[z] &= y[z] - 1u;
                uint32_t cw[W];
#pragma unroll
                for (int q = z; q < W; q++) {
                    cw[q] = y[q] & ~r[q];
                    t += __popc(cw[q]);
                }
#pragma unroll
                for (int q = z; q < W; q++) {
#pragma unroll 1
                    while (cw[q]) {
                        const uint32_t* ry = Hs + (32 * q + __ffs(cw[q]) - 1) * W;
                        cw[q] &= cw[q] - 1u;
#pragma unroll
                        for (int o = q; o < W; o++) q4 += __popc(cw[o] & ~ry[o]);
                    }
                }
            }
        }
    }
    const long long ss = (long long)s * (s - 1);
    long long v4 = 24 * q4 + 24 * b * t - 6 * b * (b - 1) * se, v3 = 24 * t - 12 * b * se;
    if (lane == 0) {
        v4 += 6 * b * (b - 1) * ss + 4 * b * (b - 1) * (b - 2) * s + b * (b - 1) * (b - 2) * (b - 3);
        v3 += 12 * b * ss + 12 * b * (b - 1) * s + 4 * b * (b - 1) * (b - 2);
    }
    c.acc[0] += v4;
    c.acc[1] += v3;
    c.acc[2] += (lane == 0 ? 12 * n * (n - 1) : 0ll) - 12 * se;
    if (lane == 0) {
        c.acc[3] += 24 * n;
        c.acc[4] += 24;
    }
    c.wops += (unsigned)(s * W);
}

// Four sizes to go: members with many non-edges are taken out one by one (each
// with the set that holds it, three sizes to go) until none has more than
// NE_SPARSE, and the rest is left to inclusion-exclusion, whose cost grows with
// the pairs of members that share non-neighbours.
template <int W>
__device__ __forceinline__ void ne_four(const NeParams& p, NeCount& c, uint32_t (&S)[W], int s, int a,
                                        const uint32_t (&h)[W][W], const uint32_t* Hs, int lane) {
    int e[W], se = 0;
    ne_degrees<W>(S, h, e, lane);
#pragma unroll
    for (int x = 0; x < W; x++) se += e[x];
    if (2 * __reduce_add_sync(GPM_FULL_MASK, (unsigned)se) > (unsigned)(s * (s - 1))) {
        ne_quads_graph<W>(p, c, S, s, a, e, h, Hs, lane);
        return;
    }
#pragma unroll 1
    while (p.k_hi - 4 + s + a >= p.k_lo) {
        int key = 0;
#pragma unroll
        for (int x = 0; x < W; x++) key = max(key, (e[x] << 7) | (32 * x + lane));
        key = (int)__reduce_max_sync(GPM_FULL_MASK, (unsigned)key);
        if ((key >> 7) <= NE_SPARSE) {
            ne_quads<W>(p, c, S, s, a, e, h, Hs, lane);
            return;
        }
        const int v = key & 127;
        uint32_t in[W], hv[W];
        int si = 0;
#pragma unroll
        for (int z = 0; z < W; z++) {
            hv[z] = Hs[v * W + z];
            if (z == (v >> 5)) S[z] &= ~(1u << (v & 31));
            in[z] = S[z] & ~hv[z];
            si += __popc(in[z]);
        }
        s--;
        if (p.k_hi - 3 + si + a >= p.k_lo) ne_triples<W, true>(p, c, in, si, a, h, Hs, lane);
#pragma unroll
        for (int x = 0; x < W; x++) {
            e[x] -= (int)((hv[x] >> lane) & 1u);
            if (!((S[x] >> lane) & 1u)) e[x] = 0;
        }
    }
}

// ne_four for the members with non-edges of a set that is small within its
// universe of 32 W members: they are re-indexed once more.  some, m: these
// members and their number (<= 32 V); idx, Hq: scratch for 64 members and
// their rows of two words.
template <int W, int V>
__device__ __forceinline__ void ne_four_again(const NeParams& p, NeCount& c, const uint32_t (&some)[W], int m, int a,
                                              const uint32_t* Hs, uint32_t* idx, uint32_t* Hq, int lane) {
    int at = 0;
#pragma unroll
    for (int x = 0; x < W; x++) {
        if ((some[x] >> lane) & 1u) idx[at + __popc(some[x] & gpm_lanemask_lt())] = 32 * x + lane;
        at += __popc(some[x]);
    }
    __syncwarp();
    // the lane's members' rows, their bits at the members closed up
    uint32_t g[V][V], T[V];
    uint32_t row[V][W];
#pragma unroll
    for (int b = 0; b < V; b++) {
        const uint32_t* r = Hs + (32 * b + lane < m ? idx[32 * b + lane] : 0u) * W;
#pragma unroll
        for (int z = 0; z < W; z++) row[b][z] = r[z];
#pragma unroll
        for (int q = 0; q < V; q++) g[b][q] = 0u;
        T[b] = m >= 32 * b + 32 ? 0xffffffffu : m <= 32 * b ? 0u : (1u << (m - 32 * b)) - 1u;
    }
    int j = 0;
#pragma unroll
    for (int z = 0; z < W; z++) {
#pragma unroll 1
        for (uint32_t y = some[z]; y; y &= y - 1u) {
            const int from = __ffs(y) - 1;
#pragma unroll
            for (int b = 0; b < V; b++) {
                const uint32_t bit = ((row[b][z] >> from) & 1u) << (j & 31);
#pragma unroll
                for (int q = 0; q < V; q++) g[b][q] |= (V == 1 || q == (j >> 5)) ? bit : 0u;
            }
            j++;
        }
    }
#pragma unroll
    for (int b = 0; b < V; b++)
#pragma unroll
        for (int q = 0; q < V; q++) {
            if (32 * b + lane >= m) g[b][q] = 0u;
            Hq[(32 * b + lane) * V + q] = g[b][q];
        }
    __syncwarp();
    ne_four<V>(p, c, T, m, a, g, Hq, lane);
    __syncwarp();
}

// All cliques of a re-indexed set of m <= 32 W members below a traversal of
// size h0 (k_hi - h0 >= 3), `a` further members being adjacent to every
// other.  Hs: m x W words, the rows of H (no diagonal); stk: the sets of the
// levels above the current one, W words at stk[W * level]; scratch: 64 + 128
// words (W > 1).  Depth first: at each level the members are taken out by
// descending number of non-edges, going down into the set that holds the one
// taken, to four sizes to go.
template <int W>
__device__ __forceinline__ void ne_sets(const NeParams& p, NeCount& c, int m, int a, int h0, const uint32_t* Hs,
                                        uint32_t* stk, uint32_t* scratch, int lane) {
    uint32_t h[W][W], S[W];
#pragma unroll
    for (int x = 0; x < W; x++) {
#pragma unroll
        for (int z = 0; z < W; z++) h[x][z] = 32 * x + lane < m ? Hs[(32 * x + lane) * W + z] : 0u;
        const int left = m - 32 * x;
        S[x] = left >= 32 ? 0xffffffffu : left <= 0 ? 0u : (1u << left) - 1u;
    }
    int lv = h0;
#pragma unroll 1
    for (;;) {
        // a set of a traversal of size lv
        int s = 0;
#pragma unroll
        for (int z = 0; z < W; z++) s += __popc(S[z]);
        // three sizes to go: at the top, or (W > 1) below a set of four that is too
        // large to be re-indexed again
        if (lv + 3 == p.k_hi) {
            ne_triples<W, false>(p, c, S, s, a, h, Hs, lane);
            if (W == 1 || lv == h0) return;
            lv--;
#pragma unroll
            for (int z = 0; z < W; z++) S[z] = stk[W * lv + z];
            __syncwarp();
            continue;
        }
        bool down = false, four = false;
        int e[W];
        ne_degrees<W>(S, h, e, lane);
        if (lv + 4 == p.k_hi) {
            if constexpr (W == 1) {
                if (lv + s + a >= p.k_lo) ne_four<1>(p, c, S, s, a, h, Hs, lane);
                four = true;
            } else {
                uint32_t some[W];
                int m4 = 0;
#pragma unroll
                for (int x = 0; x < W; x++) {
                    some[x] = __ballot_sync(GPM_FULL_MASK, e[x] > 0);
                    m4 += __popc(some[x]);
                }
                four = m4 <= 64;
                if (lv + s + a >= p.k_lo) {
                    if (m4 <= 32) ne_four_again<W, 1>(p, c, some, m4, a + s - m4, Hs, scratch, scratch + 64, lane);
                    else if (m4 <= 64) ne_four_again<W, 2>(p, c, some, m4, a + s - m4, Hs, scratch, scratch + 64, lane);
                }
            }
            ne_settle(p, c, lane);
        }
        if (!four) {
            c.wops += (unsigned)(s * W);
#pragma unroll 1
            while (lv + s + a >= p.k_lo) {
                int key = 0;
#pragma unroll
                for (int x = 0; x < W; x++) key = max(key, (e[x] << 7) | (32 * x + lane));
                key = (int)__reduce_max_sync(GPM_FULL_MASK, (unsigned)key);
                if ((key >> 7) <= 1) {
                    int one = 0;
#pragma unroll
                    for (int x = 0; x < W; x++) one += e[x];
                    const int b = (int)__reduce_add_sync(GPM_FULL_MASK, (unsigned)one) / 2;
                    ne_matching(p, c, lv, s + a, b, lane);
                    break;
                }
                const int v = key & 127;
                uint32_t in[W], hv[W];
                int si = 0;
#pragma unroll
                for (int z = 0; z < W; z++) {
                    hv[z] = Hs[v * W + z];
                    if (z == (v >> 5)) S[z] &= ~(1u << (v & 31));
                    in[z] = S[z] & ~hv[z];
                    si += __popc(in[z]);
                }
                s--;
                if (lv + 1 + si + a >= p.k_lo) {
                    if (lane == 0) {
#pragma unroll
                        for (int z = 0; z < W; z++) stk[W * lv + z] = S[z];
                    }
                    __syncwarp();
#pragma unroll
                    for (int z = 0; z < W; z++) S[z] = in[z];
                    lv++;
                    down = true;
                    break;
                }
#pragma unroll
                for (int x = 0; x < W; x++) {
                    e[x] -= (int)((hv[x] >> lane) & 1u);
                    if (!((S[x] >> lane) & 1u)) e[x] = 0;
                }
            }
        }
        if (down) continue;
        if (lv == h0) return;
        lv--;
#pragma unroll
        for (int z = 0; z < W; z++) S[z] = stk[W * lv + z];
        __syncwarp();
    }
}

}  // namespace gpm
