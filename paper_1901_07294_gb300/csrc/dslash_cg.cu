// Host side of the CG iteration's hops (dslash_cg.cuh).
#include "cg_iter.h"
#include "dslash_cg.cuh"
#include "dslash_launch.cuh"

namespace wd {

int hop_setup(const wd_gauge *g, int prec, int recon, HopArgs &A);
std::pair<int, int> hop_config(wd_ctx *ctx, const HopArgs &A, int prec, int recon, int nrhs, std::pair<int, int> def);

namespace {

// The launch shape is the context's entry for an even-odd hop of the same problem (tuned or
// pinned): its block size and, of its variant, the schedule (0 or 1) and how the links are
// loaded.  These hops have no builds of their own for schedule 2, the 3-block build (4), the
// shared-memory window (8) and two sites per thread (9), which run as schedule 1; 16-bit
// storage always runs spin-paired, schedule 0 with links loaded without L1 allocation and
// schedule 1 with it.
// Without an entry: 64 threads, links without L1 allocation, schedule 0, and 1 for FP32 with
// the axpy term (a solve, ms, schedule 0 / 1, FP32: 16^4 4.85 / 4.74, 24^3 x 48 28.5 / 28.1, 32^4 41.5
// / 41.2; 12 reals 16^4 4.80 / 4.68, 16^3 x 32 6.69 / 6.54, 24^3 x 48 24.9 / 25.0, 32^4 36.2 / 36.4; FP16,
// spin-paired, 16^4 4.32 / 4.23, 24^3 x 32 12.9 / 13.2, 24^3 x 48 19.2 / 19.9).
template <int P, int RECON, int PF, bool LNA>
cudaError_t launch_step(int step, const HopArgs &A, const CgHop &C, int threads, cudaStream_t s)
{
    const int blocks = (A.vh + threads - 1) / threads;
    const dim3 block(threads);
    if (step == CG_NORM) return wd_launch(hop_cg_kernel<P, RECON, CG_NORM, PF, LNA>, dim3(blocks), block, 0, s, A, C, 0);
    if (step == CG_RESID)
        return wd_launch(hop_cg_kernel<P, RECON, CG_RESID, PF, LNA>, dim3(blocks), block, 0, s, A, C, 0);
    const int parts = cg_parts(A.vh, threads);
    return wd_launch(hop_cg_kernel<P, RECON, CG_ALPHA, PF, LNA>, dim3(parts + blocks), block, 0, s, A, C, parts);
}

template <int P, int RECON>
cudaError_t launch_step(int step, const HopArgs &A, const CgHop &C, std::pair<int, int> cfg, cudaStream_t s)
{
    const int v = cfg.second;
    const bool first = v == 0 || v == HOP_NA0_VARIANT || v == HOP_SP0_VARIANT || v == HOP_ROW_VARIANT;   // schedule 0
    if constexpr (Prec<P>::scaled) {
        return first ? launch_step<P, RECON, 0, true>(step, A, C, cfg.first, s)
                     : launch_step<P, RECON, 1, false>(step, A, C, cfg.first, s);
    } else {
        const bool na = v == HOP_NA0_VARIANT || v == HOP_NA1_VARIANT;
        if (first) return na ? launch_step<P, RECON, 0, true>(step, A, C, cfg.first, s)
                             : launch_step<P, RECON, 0, false>(step, A, C, cfg.first, s);
        return na ? launch_step<P, RECON, 1, true>(step, A, C, cfg.first, s)
                  : launch_step<P, RECON, 1, false>(step, A, C, cfg.first, s);
    }
}

template <int P>
cudaError_t launch_step(int recon, int step, const HopArgs &A, const CgHop &C, std::pair<int, int> cfg, cudaStream_t s)
{
    return recon == 12 ? launch_step<P, 12>(step, A, C, cfg, s) : launch_step<P, 18>(step, A, C, cfg, s);
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
    const int def = prec != WD_F32 ? HOP_SP0_VARIANT : x ? HOP_NA1_VARIANT : HOP_NA0_VARIANT;
    const std::pair<int, int> cfg = hop_config(g->ctx, A, prec, recon, 1, {64, def});
    cudaError_t e;
    switch (prec) {
    case WD_F16: e = launch_step<PREC_F16>(recon, step, A, C, cfg, s); break;
    case WD_BF16: e = launch_step<PREC_BF16>(recon, step, A, C, cfg, s); break;
    default: e = launch_step<PREC_F32>(recon, step, A, C, cfg, s); break;
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
