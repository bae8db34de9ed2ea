// C entry points of the Wilson-Dirac operator: dslash_apply (full lattice)
// and dslash_eo_apply (even-odd block with fused axpby).
#include <cstdio>
#include <string>

#include "dslash_launch.cuh"
#include "wd_internal.h"

namespace wd {
extern template cudaError_t launch_hop<PREC_F64>(const HopArgs &, int, int, int, int, int, cudaStream_t);
extern template cudaError_t launch_hop<PREC_F32>(const HopArgs &, int, int, int, int, int, cudaStream_t);
extern template cudaError_t launch_hop<PREC_F16>(const HopArgs &, int, int, int, int, int, cudaStream_t);
extern template cudaError_t launch_hop<PREC_BF16>(const HopArgs &, int, int, int, int, int, cudaStream_t);
extern template cudaError_t launch_hop<PREC_DF>(const HopArgs &, int, int, int, int, int, cudaStream_t);

static bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// Key of a hop launch in the tuning cache (dagger shares its configuration).
std::string hop_key(const wd_ctx *ctx, const HopArgs &A, int prec, int recon, int nrhs)
{
    const bool hx = A.x[0] != nullptr || A.x[1] != nullptr;
    char buf[160];
    snprintf(buf, sizeof(buf), "hop sm%d p%d r%d np%d x%d n%d L%dx%dx%dx%d", ctx->num_sms, prec, recon, A.nparity,
             hx ? 1 : 0, nrhs, A.L[0], A.L[1], A.L[2], A.L[3]);
    return buf;
}

// Default shape of the shared-link kernel: {threads (mrhs_threads), variant}.
// Site order: a source spinor is read as t+ neighbour and again, 2 Lz slices
// later, as t- neighbour.  Where what is touched in between exceeds about half of L2 the
// slices are visited in the widest z-strips whose 2 w slices take no more than 0.4
// of it.  us, natural order / strips of 16 / of 8 (MB between the two reads in
// natural order; L2 129 MB): FP32 full on 32^4, 12 fields 855 / 772 / 734 (170), 6
// fields 422 / 403 / 408 (94), 4 fields 300 / 300 / 310 (69); even-odd, 12 fields 370 /
// 357 / 359 (94), 5 fields 185 / 195 / 197 (50); FP16 even-odd, 12 fields 275 / 284 / 286 (50).
static std::pair<int, int> mrhs_default(const HopArgs &A, int prec, int recon, int nrhs)
{
    const long long blocks = (long long)((A.vh + 31) / 32) * A.nparity;
    int variant = HOP_MRHS_VARIANT;
    if (prec == WD_F64) return {128, variant};   // bound by the FP64 pipe
    const int threads = mrhs_threads(blocks, nrhs, prec == WD_F32, device_sm_count());
    const double field = half_field_bytes(1, prec), link = link_block_bytes(1, link_prec(prec), recon);
    const double slice = (double)(A.L[0] / 2) * A.L[1] * A.nparity * (2 * nrhs * field + 8 / A.nparity * link);
    const double l2 = (double)device_l2_bytes();
    if (2 * A.L[2] * slice > 0.55 * l2) {
        for (int v = 5; v <= 7; ++v)   // strips of 16, 8, 4
            if (hop_mrhs_strip(v) < A.L[2] && (2 * hop_mrhs_strip(v) * slice <= 0.4 * l2 || v == 7)) {
                variant = v;
                break;
            }
    }
    return {threads, variant};
}

// Untuned defaults, from tuning runs on GB300 (8^4 to 32^4): 64-thread blocks.
// Full operator: schedule 1; with 16-bit storage and 12-real links schedule 2, which also
// prefetches the backward links, once the call touches more than three quarters of L2 and
// those links are no longer found there (FP16, us, schedule 1 / 2, without and with dagger:
// 16^3 x 32 (26 MB) 9.2 / 9.2 and 8.9 / 9.4, 24^4 (66) 22.2 / 21.7 and 21.7 / 21.9, 24^3 x 32 (88)
// 29.6 / 28.4 and 28.6 / 28.7, 32^2 x 16 x 32 (105) 34.5 / 33.0 and 33.6 / 33.4, 24^3 x 48 (133) 43.0 /
// 40.8 and 41.7 / 41.2, 32^4 (210) 64.9 / 62.0 and 63.1 / 62.6; L2 129 MB).
// Even-odd hops (each link read once) load the links without L1 allocation.  FP32: schedule
// 0, but 1 with the axpy term and 18-real links, except on grids of 7 or 8 blocks per SM,
// just under the one wave that is resident.  us, schedule 0 / 1, calls on several gauge
// fields in turn: 12^3 x 24 6.1 / 5.2, 16^4 6.6 / 6.0, 14 x 16 x 20^2 8.0 / 7.7, 16^3 x 32 (7 blocks per
// SM) 9.6 / 10.3, 20 x 26 x 6 x 44 (8) 10.2 / 10.7, 18^3 x 28 15.7 / 15.0, 20^3 x 24 17.3 / 16.5, 24^4 26.6
// / 25.6, 24^3 x 32 31.1 / 31.4, 24^3 x 40 39.1 / 38.5, 24^3 x 48 47.1 / 45.5; on one field again and
// again 16^4 4.9 / 4.7, 16^3 x 32 7.7 / 7.3, 20^3 x 24 14.3 / 12.9, 24^4 25.7 / 24.0, 24^3 x 48 47.2 / 45.7,
// 32^4 70.0 / 67.9.  Without the term 16^3 x 32 7.2 / 7.4, 24^3 x 48 43.3 / 43.6; 12 reals with it
// 16^3 x 32 6.4 / 6.5, 24^4 20.7 / 20.1, 24^3 x 48 37.3 / 37.4, 32^4 55.1 / 55.8.  16-bit: the spin-paired
// kernel (schedule 0).
// FP64 (bound by the FP64 pipe): three threads per site or one (f64_three_threads; 128: the
// block size of the latter and of an open-boundary pass, which uses hop_kernel).
static std::pair<int, int> hop_default(const HopArgs &A, int prec, int recon, int nrhs)
{
    const bool hx = A.x[0] != nullptr || A.x[1] != nullptr;
    if (prec == WD_DF) return {96, HOP_ROW_VARIANT};   // double-word: three threads per site
    if (nrhs > 1) return mrhs_default(A, prec, recon, nrhs);
    if (prec == WD_F64) {
        const long long blocks = (long long)((A.vh + 31) / 32) * A.nparity;
        return {128, f64_three_threads(blocks, device_sm_count(), recon) ? HOP_ROW_VARIANT : 0};
    }
    if (prec == WD_F32) {
        if (A.nparity == 2) return {64, 1};
        const int sms = device_sm_count(), k = ((A.vh + 63) / 64 + sms - 1) / sms;
        return {64, hx && recon == 18 && k != 7 && k != 8 ? HOP_NA1_VARIANT : HOP_NA0_VARIANT};
    }
    if (A.nparity == 1) return {64, HOP_SP0_VARIANT};
    const double bytes = 2.0 * A.vh * (2 * half_field_bytes(1, prec) + 4 * link_block_bytes(1, link_prec(prec), recon));
    return {64, recon == 12 && bytes > 0.75 * device_l2_bytes() ? 2 : 1};
}

int hop_launch_cfg(const HopArgs &A, int prec, int recon, int dagger, int nrhs, int threads, int variant,
                   cudaStream_t s)
{
    if (threads < 32 || threads > 256 || (threads & 31) || variant < 0 || variant > HOP_MAX_VARIANT)
        return set_error(WD_EINVAL, "bad hop launch configuration (%d threads, variant %d)", threads, variant);
    cudaError_t e = cudaSuccess;
    switch (prec) {
    case WD_F64: e = launch_hop<PREC_F64>(A, recon, dagger, nrhs, threads, variant, s); break;
    case WD_F32: e = launch_hop<PREC_F32>(A, recon, dagger, nrhs, threads, variant, s); break;
    case WD_F16: e = launch_hop<PREC_F16>(A, recon, dagger, nrhs, threads, variant, s); break;
    case WD_BF16: e = launch_hop<PREC_BF16>(A, recon, dagger, nrhs, threads, variant, s); break;
    case WD_DF: e = launch_hop<PREC_DF>(A, recon, dagger, nrhs, threads, variant, s); break;
    }
    if (e != cudaSuccess) return set_error(WD_ECUDA, "hop kernel launch failed: %s", cudaGetErrorString(e));
    return WD_OK;
}

// {threads, variant} of a hop: the context's entry for its shape, else `def`.
std::pair<int, int> hop_config(wd_ctx *ctx, const HopArgs &A, int prec, int recon, int nrhs, std::pair<int, int> def)
{
    // the key of a launch is a string: 1 us to build, on a call of 3 us
    if (!ctx->any_tuned.load(std::memory_order_acquire)) return def;
    return tuned_config(ctx, hop_key(ctx, A, prec, recon, nrhs), def);
}

int hop_launch(wd_ctx *ctx, const HopArgs &A, int prec, int recon, int dagger, int nrhs, cudaStream_t s)
{
    const auto cfg = hop_config(ctx, A, prec, recon, nrhs, hop_default(A, prec, recon, nrhs));
    return hop_launch_cfg(A, prec, recon, dagger, nrhs, cfg.first, cfg.second, s);
}

// Fills the geometry and gauge parts of HopArgs.
int hop_setup(const wd_gauge *g, int prec, int recon, HopArgs &A)
{
    if (!g) return set_error(WD_EINVAL, "gauge is NULL");
    if (!valid_field_prec(prec)) return set_error(WD_EINVAL, "bad precision %d", prec);
    if (!valid_recon(recon)) return set_error(WD_EINVAL, "bad reconstruction %d", recon);
    const char *base = nullptr;
    WD_TRY(gauge_layout(g, prec, recon, &base));
    const int vh = g->geo.Vh;
    A.link_blk = link_block_bytes(vh, link_prec(prec), recon);
    A.gauge[0] = base;
    A.gauge[1] = base + 4 * A.link_blk;
    for (int mu = 0; mu < 4; ++mu) A.L[mu] = g->geo.L[mu];
    A.vh = vh;
    A.tneg = g->t_sign < 0 ? 1 : 0;
    A.status = ctx_status_word(g->ctx);
    div_magic((unsigned)(A.L[0] >> 1), A.div_m[0], A.div_s[0]);
    div_magic((unsigned)A.L[1], A.div_m[1], A.div_s[1]);
    div_magic((unsigned)A.L[2], A.div_m[2], A.div_s[2]);
    return WD_OK;
}

int eo_hop(const wd_gauge *g, int prec, int recon, void *out, const void *in, const void *x, int p, double a,
           double b, int dagger, cudaStream_t s, bool beside)
{
    HopArgs A{};
    A.beside = beside;
    WD_TRY(hop_setup(g, prec, recon, A));
    A.in[0] = A.in[1] = (const char *)in;
    A.x[0] = A.x[1] = (const char *)x;
    A.out[0] = A.out[1] = (char *)out;
    A.rhs_stride = half_field_bytes(A.vh, prec);
    A.nparity = 1;
    A.parity0 = p;
    A.a = a;
    A.b = b;
    return hop_launch(g->ctx, A, prec, recon, dagger ? 1 : 0, 1, s);
}

int full_hop(const wd_gauge *g, int prec, int recon, void *out, const void *in, double a, double b, cudaStream_t s)
{
    HopArgs A{};
    WD_TRY(hop_setup(g, prec, recon, A));
    const size_t half = half_field_bytes(A.vh, prec);
    for (int p = 0; p < 2; ++p) {
        A.in[p] = (const char *)in + (size_t)(1 - p) * half;
        A.x[p] = (const char *)in + (size_t)p * half;
        A.out[p] = (char *)out + (size_t)p * half;
    }
    A.rhs_stride = 2 * half;
    A.nparity = 2;
    A.parity0 = 0;
    A.a = a;
    A.b = b;
    return hop_launch(g->ctx, A, prec, recon, 0, 1, s);
}

} // namespace wd

using namespace wd;

extern "C" {

static int full_apply(wd_ctx *ctx, const wd_gauge *g, void *out, const void *in, double mass, int dagger, int nrhs,
                      int prec, int recon, void *stream)
{
    clear_error();
    if (!ctx) return set_error(WD_EINVAL, "ctx is NULL");
    if (!out || !in) return set_error(WD_EINVAL, "NULL field pointer");
    if (!aligned16(out) || !aligned16(in)) return set_error(WD_EINVAL, "field pointers must be 16-byte aligned");
    if (out == in) return set_error(WD_EINVAL, "out must not alias in");
    if (nrhs < 1) return set_error(WD_EINVAL, "nrhs = %d must be >= 1", nrhs);
    HopArgs A{};
    WD_TRY(hop_setup(g, prec, recon, A));
    const size_t half = half_field_bytes(A.vh, prec);
    const char *src = (const char *)in;
    char *dst = (char *)out;
    for (int p = 0; p < 2; ++p) {
        A.in[p] = src + (size_t)(1 - p) * half;
        A.x[p] = src + (size_t)p * half;
        A.out[p] = dst + (size_t)p * half;
    }
    A.rhs_stride = 2 * half;
    A.nparity = 2;
    A.parity0 = 0;
    A.a = mass + 4.0;
    A.b = -0.5;
    return hop_launch(ctx, A, prec, recon, dagger, nrhs, (cudaStream_t)stream);
}

int dslash_apply(wd_ctx *ctx, const wd_gauge *g, void *out, const void *in, double mass, int nrhs, int prec,
                 int recon, void *stream)
{
    return full_apply(ctx, g, out, in, mass, 0, nrhs, prec, recon, stream);
}

int dslash_apply_dagger(wd_ctx *ctx, const wd_gauge *g, void *out, const void *in, double mass, int nrhs, int prec,
                        int recon, void *stream)
{
    return full_apply(ctx, g, out, in, mass, 1, nrhs, prec, recon, stream);
}

int dslash_eo_apply(wd_ctx *ctx, const wd_gauge *g, void *out, const void *in, const void *x, int out_parity,
                    double a, double b, int dagger, int nrhs, int prec, int recon, void *stream)
{
    clear_error();
    if (!ctx) return set_error(WD_EINVAL, "ctx is NULL");
    if (!out || !in) return set_error(WD_EINVAL, "NULL field pointer");
    if (!aligned16(out) || !aligned16(in) || (x && !aligned16(x)))
        return set_error(WD_EINVAL, "field pointers must be 16-byte aligned");
    if (out == in) return set_error(WD_EINVAL, "out must not alias in");
    if (out_parity != WD_EVEN && out_parity != WD_ODD) return set_error(WD_EINVAL, "out_parity must be 0 or 1");
    if (nrhs < 1) return set_error(WD_EINVAL, "nrhs = %d must be >= 1", nrhs);
    HopArgs A{};
    WD_TRY(hop_setup(g, prec, recon, A));
    const int p = out_parity;
    A.in[p] = A.in[1 - p] = (const char *)in;
    A.x[p] = A.x[1 - p] = (const char *)x;
    A.out[p] = A.out[1 - p] = (char *)out;
    A.rhs_stride = half_field_bytes(A.vh, prec);
    A.nparity = 1;
    A.parity0 = p;
    A.a = a;
    A.b = b;
    return hop_launch(ctx, A, prec, recon, dagger ? 1 : 0, nrhs, (cudaStream_t)stream);
}

} // extern "C"
