// motif_hom.cuh -- induced motif counts of k = 3 .. 5 vertices from
// homomorphism counts (shared by motif_hom.cu and the batched launch).
#pragma once

#include "common.cuh"

namespace gpm {

// The connected graphs on at most five vertices, by the sums that count their
// homomorphisms into G (edges 1-2, 1-3, ...: see hom_edges() in motif_hom.cu).
enum Hom {
    // d^a s^b T^c summed over the vertices u: d = degree of u, s = sum of its
    // neighbours' degrees, T = twice its triangles
    H_POINT, H_EDGE, H_CHERRY, H_TRI, H_STAR3, H_PATH4, H_PAW, H_STAR4, H_PATH5, H_FORK, H_CRICKET, H_LOLLI, H_BOWTIE,
    H_UNIFORM,                         // their number
    // the rest: sums over pairs and triples of vertices
    H_CYCLE4 = H_UNIFORM, H_DIAMOND, H_K4, H_CYCLE5, H_BANNER, H_BULL, H_K23, H_DART, H_KITE, H_HOUSE, H_GEM, H_BOOK,
    H_K4TAIL, H_SPOKE, H_WHEEL, H_K5P3, H_K5E, H_K5, HOM_N
};

// Counts of size k from the sums: pattern p occurs
// (sum_j coef[p * HOM_N + j] hom[j]) / aut[p] times (wrapping 64-bit sums, the
// result of which is exact: every homomorphism count is below 2^63).
struct HomTable {
    int k = 0, npat = 0;
    std::vector<long long> coef;
    std::vector<long long> aut;
};
const HomTable& hom_table(int k);                 // host, built once per k
void hom_combine(const HomTable& t, const unsigned long long* hom, uint64_t* counts_out);
const long long* device_hom_table(int k, cudaStream_t s);   // coef, then aut; uploaded once per device, on s

struct HomLaunch {
    const int32_t* __restrict__ indptr;
    const int32_t* __restrict__ indices;
    const int32_t* __restrict__ deg;
    const int32_t* __restrict__ goff;     // batch: vertex range of every graph (nullptr: one graph)
    const int32_t* __restrict__ vgraph;   // batch: graph of every vertex
    const uint32_t* __restrict__ edges;   // k = 5: ensure_hom_edges
    long long n;
    int parts;                            // warps that share a vertex
    int grab;                             // parts a warp takes at a time
    int maxn;                             // vertices of the largest graph
    int maxd;                             // largest degree
    int warp_words, m_words;              // shared words per warp, those of its bit sets
    unsigned long long* hom;              // [graph][HOM_N], zero
    unsigned long long* ticket;           // next vertex, zero
    Control* ctl;
    unsigned long long* busy;             // this launch's warp time
};

constexpr int HOM_WARPS = 4;              // warps per block
constexpr int HOM_MAX_N = 16384;          // vertices of one graph (shared-memory arrays over them)
constexpr int HOM_MAX_D = 1024;           // largest degree (bit rows over a neighbourhood)
// k = 3, 4: with a larger degree than this the edge sums are faster (one warp
// has the largest vertex).  R-MAT, whole call, these / edge sums, k = 4: degree 74
// 74 / 78 us, 123 110 / 93, 931 6,400 / 230; block-model graph, degree 100: 200 /
// 250; k = 3: degree 123 53 / 77, 216 82 / 80, 931 450 / 155.
constexpr int HOM_HUB_D3 = 210, HOM_HUB_D4 = 110;
// And with more vertices than this, whose arrays leave few warps resident.
// Random graphs of average degree 6 / 16 / 60, these and edge sums in us: k = 3,
// n = 4,000: 58, 65 / 60, 74 / 85, 152; 8,000: 60, 73 / 64, 71 / 136, 160; 12,000:
// 74, 67 / 86, 72 / 238, 188; 16,384: 116, 71 / 146, 75 / 534, 216; k = 4, n = 4,000:
// 64, 120 / 84, 136 / 384, 265; 6,000: 71, 142 / 111, 179 / 521, 383; 8,000: 127, 174 /
// 200, 191 / 1,218, 413; 16,384: 371, 206 / 632, 244 / 4,525, 686.
constexpr int HOM_SUMS_N3 = 8192, HOM_SUMS_N4 = 6144;

// Whether graphs of at most n vertices and degree d are counted this way.
bool hom_applies(long long n, long long d, int k);
int hom_warp_words(int n, int d, int k);
int hom_m_words(int n, int d);
// The edge list of k = 5 (kept with the graph); goff, vgraph: the batch's, or null.
const uint32_t* ensure_hom_edges(gpm_graph* g, const int32_t* goff, const int32_t* vgraph);
// Fills warp_words and sizes the launch (no stream operations); the launch itself (nothing
// throws between the two ends of a capture).
Grid plan_hom(HomLaunch& p, int k, int sms, const gpm_config& cfg);
cudaError_t launch_hom(const HomLaunch& p, int k, const Grid& gr, cudaStream_t s);
// Whole-graph counts of g where hom_applies (stats filled)
void run_motif_hom(gpm_graph* g, int k, uint64_t* counts_out);
// Larger graphs, k = 3 and 4 (motif_sparse.cu; builds the orientation)
bool motif_sparse_applies(gpm_graph* g, int k);
void run_motif_sparse(gpm_graph* g, int k, uint64_t* counts_out);
// out[g * npat + p] = count of pattern p in graph g; clique_k > 0 (at most k): the
// cliques of that size of every graph as well, from the same sums
cudaError_t launch_hom_finish(const unsigned long long* hom, int n_graphs, int k, unsigned long long* out, int clique_k,
                              unsigned long long* clique_out, cudaStream_t s);

}  // namespace gpm
