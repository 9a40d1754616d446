// k_hom<5> (motif_hom.cu) on the CPU over one graph: argv[1] names a file of
// int32 n, indptr[n + 1], indices[].  A write outside of its shared memory
// ends the run; else the sums are printed.
#include "simt.h"
#include "device_part.h"

namespace gpm {
DevBuf::~DevBuf() {}
}
using namespace gpm;

int main(int argc, char** argv) {
    std::vector<int32_t> in(1 << 20);
    FILE* f = argc > 1 ? fopen(argv[1], "rb") : nullptr;
    if (!f) return 1;
    in.resize(fread(in.data(), 4, in.size(), f));
    fclose(f);
    const int n = in[0];
    std::vector<int32_t> deg(n);
    std::vector<uint32_t> edges;
    HomLaunch p{};
    p.indptr = &in[1];
    p.indices = &in[n + 2];
    for (int v = 0; v < n; v++) {
        deg[v] = p.indptr[v + 1] - p.indptr[v];
        p.maxd = max(p.maxd, deg[v]);
        for (int q = p.indptr[v]; q < p.indptr[v + 1]; q++) edges.push_back((uint32_t)v << 16 | (uint32_t)p.indices[q]);
    }
    Control ctl{};
    std::vector<unsigned long long> hom(HOM_N, 0);
    p.deg = deg.data();
    p.edges = edges.data();
    p.n = p.maxn = n;
    p.parts = 2;
    p.grab = 1;
    p.warp_words = hom_warp_words(n, p.maxd, 5);
    p.m_words = min(hom_m_words(n, p.maxd), 3 * ((p.maxd + 31) / 32));   // three vertices a range
    p.hom = hom.data();
    p.ticket = &ctl.next_root;
    p.ctl = &ctl;
    simt_run(32, p.warp_words, [&] { k_hom<5>(p); });
    for (unsigned long long h : hom) printf("%llu ", h);
}
