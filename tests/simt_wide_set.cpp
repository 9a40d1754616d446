// The sets of one root's child (ne_child, clique_nonedge.cu) on the CPU: a
// candidate set of 66 disjoint non-edges and three hubs, each non-adjacent to
// half of the others.  The hubs are taken out one by one, the set that holds
// each has three sizes to go, and what is left is counted as a matching.
// argv[1]: what every lane holds in acc[0] from the root's earlier sets.  Prints
// the largest |acc[0]| over the lanes afterwards, the cliques counted once all
// is folded, and the set's 4-cliques.
#include "simt.h"
#include "device_part.h"

namespace gpm {
DevBuf::~DevBuf() {}
}
using namespace gpm;

int main(int argc, char** argv) {
    if (argc < 2) return 1;
    const long long before = atoll(argv[1]);
    const int pairs = 66, hubs = 3, d = 2 * pairs + hubs;
    NeLaunch p{};
    p.ne.k_lo = p.ne.k_hi = 6;
    p.maxd = d;
    p.w = (d + 31) / 32;
    p.ws = p.w | 1;
    std::vector<unsigned long long> binom((size_t)(NE_BINOM_N + 1) * NE_BINOM_K, 0ull);
    for (int n = 0; n <= d; n++)
        for (int k = 0; k < NE_BINOM_K; k++)
            binom[n * NE_BINOM_K + k] = k == 0 ? 1 : n == 0 ? 0 : binom[(n - 1) * NE_BINOM_K + k - 1] + binom[(n - 1) * NE_BINOM_K + k];
    p.ne.binom = binom.data();
    std::vector<uint32_t> rows((size_t)d * p.ws, 0u);
    std::vector<std::vector<char>> adj(d, std::vector<char>(d, 0));
    for (int i = 0; i < d; i++)
        for (int j = i + 1; j < d; j++) {
            const bool non = j < 2 * pairs ? i % 2 == 0 && j == i + 1 : i < 2 * pairs && (i / 2 + j) % 2 == 0;
            if (non) continue;
            adj[i][j] = adj[j][i] = 1;
            rows[i * p.ws + (j >> 5)] |= 1u << (j & 31);
            rows[j * p.ws + (i >> 5)] |= 1u << (i & 31);
        }
    long long most = 0;
    unsigned long long counted = 0, want = 0;
    simt_run(32, ne_warp_words(d, p.w, true), [&] {
        const int lane = threadIdx.x, dpad = (d + 3) & ~3;
        NeWarp k;
        k.cand = simt_smem;
        k.Hs = k.cand + NE_LEVELS * p.w;
        k.stk = k.Hs + 32 * NE_W * NE_W;
        k.scratch = k.stk + NE_W * NE_LEVELS;
        k.mem = reinterpret_cast<uint16_t*>(k.scratch + NE_SCRATCH);
        k.wide = k.mem + dpad;
        k.we = k.wide + dpad;
        if (lane < p.w) k.cand[2 * p.w + lane] = lane < d / 32 ? ~0u : (1u << (d % 32)) - 1u;
        __syncwarp();
        NeCount c;
        c.acc[0] = before;
        ne_child<true>(p, c, k, rows.data(), p.w, lane);
        most = max(most, c.acc[0] < 0 ? -c.acc[0] : c.acc[0]);
        ne_fold(p.ne, c, lane);
        if (lane == 6) counted = c.size;
        if (c.ovf) abort();
    });
    // 4-cliques of the set
    for (int a = 0; a < d; a++)
        for (int b = a + 1; b < d; b++)
            if (adj[a][b])
                for (int e = b + 1; e < d; e++)
                    if (adj[a][e] && adj[b][e])
                        for (int f = e + 1; f < d; f++) want += adj[a][f] && adj[b][f] && adj[e][f];
    printf("%lld %llu %llu\n", most, counted, want);
}
