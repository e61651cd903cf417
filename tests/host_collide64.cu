// Host build of the FP64 collisions of lbm_collide64.cuh, for the CPU test
// that compares them with the oracle: one node's stored deviations in and out
// in the kernel's population order.  Test infrastructure only.
#include "../paper_2212_07494_gb300/csrc/lbm_collide64.cuh"

using namespace lbm;

namespace {
template <int L> int run(int trim, const double *din, const double *g, double om2, double *dout) {
    double G[Grid<Lat<L>::D>::N] = {0.0};
    for (int i = 0; i < Lat<L>::Q; ++i) G[gpos<L>(i)] = din[i];
    if (trim && L != D2Q9) return -1;
    if (trim) collide_smrt_trim64(G, g[0], g[1], om2);
    else collide_bgk64<L>(G, g[0], g[1], Lat<L>::D == 3 ? g[2] : 0.0, om2);
    for (int i = 0; i < Lat<L>::Q; ++i) dout[i] = G[gpos<L>(i)];
    return 0;
}
}  // namespace

extern "C" int host_collide64(int lat, int trim, const double *din, const double *g, double tau2, double *dout) {
    return lat == D2Q9 ? run<D2Q9>(trim, din, g, 1.0 / tau2, dout)
         : lat == D3Q19 ? run<D3Q19>(trim, din, g, 1.0 / tau2, dout)
                        : run<D3Q27>(trim, din, g, 1.0 / tau2, dout);
}
