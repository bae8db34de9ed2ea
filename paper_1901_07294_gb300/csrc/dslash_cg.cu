// Host side of the CG iteration's hops (dslash_cg.cuh).
#include "cg_iter.h"
#include "dslash_cg.cuh"

namespace wd {

int hop_setup(const wd_gauge *g, int prec, int recon, HopArgs &A);

namespace {

constexpr int CG_HOP_THREADS = 64;   // the untuned hops' block size

template <int P, int RECON> cudaError_t launch_step(int step, const HopArgs &A, const CgHop &C, cudaStream_t s)
{
    const int blocks = (A.vh + CG_HOP_THREADS - 1) / CG_HOP_THREADS;
    const dim3 block(CG_HOP_THREADS);
    if (step == CG_NORM) return wd_launch(hop_cg_kernel<P, RECON, CG_NORM>, dim3(blocks), block, 0, s, A, C, 0);
    if (step == CG_RESID) return wd_launch(hop_cg_kernel<P, RECON, CG_RESID>, dim3(blocks), block, 0, s, A, C, 0);
    const int parts = cg_parts(A.vh, CG_HOP_THREADS);
    return wd_launch(hop_cg_kernel<P, RECON, CG_ALPHA>, dim3(parts + blocks), block, 0, s, A, C, parts);
}

template <int P> cudaError_t launch_step(int recon, int step, const HopArgs &A, const CgHop &C, cudaStream_t s)
{
    return recon == 12 ? launch_step<P, 12>(step, A, C, s) : launch_step<P, 18>(step, A, C, s);
}

int cg_hop(const wd_gauge *g, int prec, int recon, int step, const char *in, const char *x, char *out, double a,
           double b, const CgHop &C, cudaStream_t s)
{
    HopArgs A{};
    WD_TRY(hop_setup(g, prec, recon, A));
    A.in[0] = A.in[1] = in;
    A.x[0] = A.x[1] = x;
    A.out[0] = A.out[1] = out;
    A.nparity = 1;
    A.parity0 = step == CG_ALPHA ? WD_ODD : WD_EVEN;
    A.a = a;
    A.b = b;
    cudaError_t e;
    switch (prec) {
    case WD_F16: e = launch_step<PREC_F16>(recon, step, A, C, s); break;
    case WD_BF16: e = launch_step<PREC_BF16>(recon, step, A, C, s); break;
    default: e = launch_step<PREC_F32>(recon, step, A, C, s); break;
    }
    if (e != cudaSuccess) return set_error(WD_ECUDA, "hop kernel launch failed: %s", cudaGetErrorString(e));
    return WD_OK;
}

} // namespace

int cg_iteration_hops(const wd_gauge *g, int prec, int recon, double mass, const CgFields &f, cudaStream_t s)
{
    const double a = mass + 4.0, c = 1.0 / (4.0 * (mass + 4.0));
    const CgHop C{f.r, f.site, f.s, RedScratch{f.partials, f.ticket}};
    WD_TRY(eo_hop(g, prec, recon, f.t_o, f.p, nullptr, WD_ODD, 0.0, 1.0, 0, s));              // H_oe p
    WD_TRY(cg_hop(g, prec, recon, CG_NORM, f.t_o, f.p, f.t_e, a, -c, C, s));                  // Mhat p
    WD_TRY(cg_hop(g, prec, recon, CG_ALPHA, f.t_e, nullptr, f.t_o, 0.0, 1.0, C, s));          // g5 H_oe g5 t
    return cg_hop(g, prec, recon, CG_RESID, f.t_o, f.t_e, nullptr, a, -c, C, s);              // r -= alpha Mhat^dagger t
}

} // namespace wd
