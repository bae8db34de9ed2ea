// BLAS-1 on device fields with deterministic FP64 reductions.
//
// One thread per site (grid-stride).  A site's 24 reals are combined in the
// compute type of the field (FP32 for the 16/32-bit formats), each site's
// contribution is added in FP64, then a fixed-order FP64 sum over the block
// (block_sum), per-block partials in scratch memory, and the
// last block to finish (atomic ticket) sums the partials the same way (thread
// t takes partials t, t+256, ...), so the order is fixed.  The
// grid size depends only on the field size, the SM count and the kernel, so
// repeated calls give bitwise identical results.
#pragma once

#include <type_traits>

#include "wd_device.cuh"

namespace wd {

constexpr int BLAS_THREADS = 256;
constexpr int MAX_RED_BLOCKS = 2048;
constexpr int MAX_NR = 4;

// Scratch used by one reduction: MAX_RED_BLOCKS*MAX_NR partials + a ticket.
struct RedScratch {
    double *partials;
    unsigned *ticket;
};

// A field seen as `nhalf` consecutive half fields of vh sites each.
template <int P> struct FieldRef {
    char *p;
    size_t half_bytes;
    int vh;
    __device__ __forceinline__ void load(int j, typename Prec<P>::real (&v)[24]) const
    {
        const int h = j >= vh;
        Spinor<P>::load(p + h * half_bytes, vh, j - h * vh, v);
    }
    __device__ __forceinline__ void store(int j, const typename Prec<P>::real (&v)[24]) const
    {
        const int h = j >= vh;
        Spinor<P>::store(p + h * half_bytes, vh, j - h * vh, v);
    }
};

// An operation without a reduction on fields of one unscaled layout can run over
// the fields' 16-byte vectors (Op::FLAT of them per site) instead of over sites: a
// thread then holds 8 registers of data instead of 96.  FP64 axpby, half fields,
// us at the start / with one form of its arithmetic issued (OpAxpby) / over
// vectors: 24^3 x 48 51.0 / 35.4 / 33.9, 32^4 72.5 / 53.2 / 52.8, 16^4 6.1 / 5.0 / 4.9,
// 8^4 5.7 / 5.1 / 1.6.  (FP32, double-word and the FP64 inner product were no faster.)
template <typename Op, typename = void> constexpr int flat_vectors = 0;
template <typename Op> constexpr int flat_vectors<Op, std::void_t<decltype(Op::FLAT)>> = Op::FLAT;

// Block sums of NR values per thread, in FP64 and in a fixed order; the sums are
// valid in thread 0.  GB300's FP64 pipe takes 16 cycles per warp instruction,
// so the sum is laid out for few of them: every thread's values go to shared
// memory, one warp adds the block's 8 values per lane and folds its 32 lanes
// (12 warp additions per value).  Folding every warp with shuffles and then
// the warps in one thread takes 48.  24^3 x 48 half fields, FP16 storage:
// inner product (NR = 2) 14.7 -> 9.1 us, norm (NR = 1) 9.4 -> 5.9 us (with
// blas_grid_for's 4 blocks per SM 8.4 and 5.8 us).
template <int NR> __device__ __forceinline__ void block_sum(double (&v)[NR], double (*sm)[BLAS_THREADS])
{
#pragma unroll
    for (int k = 0; k < NR; ++k) sm[k][threadIdx.x] = v[k];
    __syncthreads();
    if (threadIdx.x < 32) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            v[k] = sm[k][threadIdx.x];
#pragma unroll
            for (int w = 1; w < BLAS_THREADS / 32; ++w) v[k] += sm[k][threadIdx.x + 32 * w];
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
#pragma unroll
            for (int k = 0; k < NR; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
    }
}

// Takes the next ticket: this thread's earlier writes are visible to whoever
// takes a later one, and the writes of all earlier takers to this thread (and,
// after the next barrier, to its block).
__device__ __forceinline__ unsigned ticket_take(unsigned *ticket)
{
    unsigned t;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(ticket) : "memory");
    return t;
}

// The site loop and the deterministic reduction of one BLAS operation over a
// grid of blocks along x (shared by blas_kernel and the per-member kernels of
// a request group, which run one operation per blockIdx.y).
template <typename Op> __device__ __forceinline__ void blas_body(const Op &op, const int nsite, const RedScratch &rs)
{
    constexpr int NR = Op::NR;
    double acc[NR > 0 ? NR : 1];
#pragma unroll
    for (int k = 0; k < (NR > 0 ? NR : 1); ++k) acc[k] = 0.0;
    if constexpr (flat_vectors<Op> > 0) {
        // four vectors per pass, all loaded before the first is used
        const size_t n = (size_t)nsite * flat_vectors<Op>, stride = (size_t)gridDim.x * blockDim.x;
        size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
        for (; k + 3 * stride < n; k += 4 * stride) {
            typename Op::In in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) in[u] = op.vload(k + u * stride);
#pragma unroll
            for (int u = 0; u < 4; ++u) op.vuse(k + u * stride, in[u]);
        }
        for (; k < n; k += stride) op.vuse(k, op.vload(k));
    } else {
        // two sites per pass where the loop runs twice or more: the second site's
        // loads can then be in flight with the first's
        const int stride = gridDim.x * blockDim.x;
        int j = blockIdx.x * blockDim.x + threadIdx.x;
        for (; j + stride < nsite; j += 2 * stride) {
            op.site(j, acc);
            op.site(j + stride, acc);
        }
        if (j < nsite) op.site(j, acc);
    }
    if constexpr (NR > 0) {
        __shared__ double sm[NR][BLAS_THREADS];
        __shared__ bool last;
        block_sum<NR>(acc, sm);
        if (threadIdx.x == 0) {
#pragma unroll
            for (int k = 0; k < NR; ++k) rs.partials[blockIdx.x * NR + k] = acc[k];
            last = ticket_take(rs.ticket) == gridDim.x - 1;
        }
        __syncthreads();
        if (last) {   // block-uniform: the whole last block sums the partials
            double s[NR];
#pragma unroll
            for (int k = 0; k < NR; ++k) s[k] = 0.0;
            for (int b = threadIdx.x; b < (int)gridDim.x; b += BLAS_THREADS)
#pragma unroll
                for (int k = 0; k < NR; ++k) s[k] += __ldcg(rs.partials + b * NR + k);
            block_sum<NR>(s, sm);
            if (threadIdx.x == 0) {
                op.finish(s);
                *rs.ticket = 0u;   // ready for the next reduction
            }
        }
    }
}

template <typename Op>
__global__ void __launch_bounds__(BLAS_THREADS) blas_kernel(const Op op, const int nsite, const RedScratch rs)
{
    grid_dependency_enter();
    blas_body(op, nsite, rs);
}

// ---- operations -----------------------------------------------------------
// |x|^2
template <int P> struct OpNorm2 {
    static constexpr int NR = 1;
    FieldRef<P> x;
    double *out;
    __device__ __forceinline__ void site(int j, double (&a)[1]) const
    {
        typename Prec<P>::real v[24];
        x.load(j, v);
        typename Prec<P>::real s = 0;
#pragma unroll
        for (int k = 0; k < 24; ++k) s = fma(v[k], v[k], s);
        a[0] += to_real<double>(s);
    }
    __device__ __forceinline__ void finish(const double (&s)[1]) const { out[0] = s[0]; }
};

// <a, b> = sum conj(a) b  (re, im)
template <int PA, int PB> struct OpDot {
    static constexpr int NR = 2;
    FieldRef<PA> a;
    FieldRef<PB> b;
    double *out;
    __device__ __forceinline__ void site(int j, double (&acc)[2]) const
    {
        using T = typename Prec<PA>::real;
        T u[24];
        typename Prec<PB>::real w[24];
        a.load(j, u);
        b.load(j, w);
        T re = 0, im = 0;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            re = fma(u[2 * k], to_real<T>(w[2 * k]), re);
            re = fma(u[2 * k + 1], to_real<T>(w[2 * k + 1]), re);
            im = fma(u[2 * k], to_real<T>(w[2 * k + 1]), im);
            im = fma(-u[2 * k + 1], to_real<T>(w[2 * k]), im);
        }
        acc[0] += to_real<double>(re);
        acc[1] += to_real<double>(im);
    }
    __device__ __forceinline__ void finish(const double (&s)[2]) const { out[0] = s[0]; out[1] = s[1]; }
};

// Re <p, q>; also alpha = num / Re<p,q> (CG step length) into out[1].
template <int P> struct OpDotReAlpha {
    static constexpr int NR = 1;
    FieldRef<P> p, q;
    double num;
    double *out;   // out[0] = Re<p,q>, out[1] = num / out[0]
    __device__ __forceinline__ void site(int j, double (&acc)[1]) const
    {
        typename Prec<P>::real u[24], w[24];
        p.load(j, u);
        q.load(j, w);
        typename Prec<P>::real s = 0;
#pragma unroll
        for (int k = 0; k < 24; ++k) s = fma(u[k], w[k], s);
        acc[0] += to_real<double>(s);
    }
    __device__ __forceinline__ void finish(const double (&s)[1]) const
    {
        out[0] = s[0];
        out[1] = num / s[0];
    }
};

// CG update with alpha read from device memory:
//   r -= alpha * Ap;  x += alpha * p;  returns |r|^2.   x may have another precision.
template <int PX, int PR> struct OpCgUpdate {
    static constexpr int NR = 1;
    FieldRef<PX> x;
    FieldRef<PR> r, p, ap;
    const double *alpha;
    double *out;
    __device__ __forceinline__ void site(int j, double (&acc)[1]) const
    {
        using T = typename Prec<PR>::real;
        using TX = typename Prec<PX>::real;
        const double al = *alpha;
        T rv[24], pv[24], av[24];
        TX xv[24];
        r.load(j, rv);
        ap.load(j, av);
        const T a = (T)al;
        T s = 0;
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            rv[k] = fma(-a, av[k], rv[k]);
            s = fma(rv[k], rv[k], s);
        }
        r.store(j, rv);
        p.load(j, pv);
        x.load(j, xv);
        const TX ax = (TX)al;
#pragma unroll
        for (int k = 0; k < 24; ++k) xv[k] = fma(ax, to_real<TX>(pv[k]), xv[k]);
        x.store(j, xv);
        acc[0] += to_real<double>(s);
    }
    __device__ __forceinline__ void finish(const double (&s)[1]) const { out[0] = s[0]; }
};

// r = b - y; returns |r|^2 (the full solve's residuals, FP64).
template <int P> struct OpXmyNorm {
    static constexpr int NR = 1;
    FieldRef<P> b;
    FieldRef<P> y;
    FieldRef<P> r;
    double *out;
    __device__ __forceinline__ void site(int j, double (&acc)[1]) const
    {
        using T = typename Prec<P>::real;
        T bv[24];
        typename Prec<P>::real yv[24];
        b.load(j, bv);
        y.load(j, yv);
        T s = 0;
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            bv[k] -= to_real<T>(yv[k]);
            s = fma(bv[k], bv[k], s);
        }
        r.store(j, bv);
        acc[0] += to_real<double>(s);
    }
    __device__ __forceinline__ void finish(const double (&s)[1]) const { out[0] = s[0]; }
};

// r = b - y in FP64 (y may be a double-word field, widened exactly), |r|^2 from the
// FP64 values, r stored in the precision PS of the iteration it restarts.  One pass
// where storing r in FP64 and converting it took two: 58 + 17 -> 62 us on 24^3 x 48
// (double-word y, FP16 r).  Bound by the FP64 pipe (three instructions per real: 38
// us); with the conversion to FP32 on that pipe too it took 74 us (FP64 y: 55 ->
// 43 us).  The whole FP16 CG there: 19.78 -> 19.62 ms.
template <int PY, int PS> struct OpResidual {
    static constexpr int NR = 1;
    FieldRef<PREC_F64> b;
    FieldRef<PY> y;
    FieldRef<PS> r;
    double *out;
    __device__ __forceinline__ void site(int j, double (&acc)[1]) const
    {
        typename Prec<PS>::real v[24];
        double s = 0;
        const int h = j >= b.vh, i = j - h * b.vh;
#pragma unroll
        for (int k = 0; k < 12; ++k) {   // planes of two reals, the same in both formats
            const size_t o = h * b.half_bytes + ((size_t)k * b.vh + i) * 16;
            double d[2];
            typename Prec<PY>::real yv[2];
            unpack16<PREC_F64>(ldg16(b.p + o), d, 1.0f);
            unpack16<PY>(ldg16(y.p + o), yv, 1.0f);
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                d[l] -= to_real<double>(yv[l]);
                s = fma(d[l], d[l], s);
                if constexpr (PS == PREC_F64) v[2 * k + l] = d[l];
                else v[2 * k + l] = f64_to_f32(d[l]);
            }
        }
        r.store(j, v);
        acc[0] += s;
    }
    __device__ __forceinline__ void finish(const double (&s)[1]) const { out[0] = s[0]; }
};

// ---- vector updates of the mixed-precision CG iteration ----------------------
// x += alpha p, then p = r + beta p: the vector updates left to a kernel of their
// own when the hops carry the rest (dslash_cg.cuh).  alpha is read from device
// memory, beta too unless beta_dev is NULL.  x, an FP32 half field, is not touched
// again in the iteration and is read and written with streaming hints: the links and
// p stay in L2 for the next hop instead (FP16 CG on 24^3 x 48 19.79 -> 19.58 ms,
// 32^4 28.55 -> 28.42, FP32 41.87 -> 41.70; lattices that fit in L2 and request
// groups within the runs' spread).
template <int P> struct OpXp {
    static constexpr int NR = 0;
    FieldRef<PREC_F32> x;
    FieldRef<P> r, p;
    const double *alpha, *beta_dev;
    double beta;
    __device__ __forceinline__ void site(int j, double (&)[1]) const
    {
        const float al = (float)*alpha, be = (float)(beta_dev ? *beta_dev : beta);
        float rv[24], pv[24], xv[24];
        p.load(j, pv);
        uint4 *xp = reinterpret_cast<uint4 *>(x.p) + j;   // six planes of four reals
#pragma unroll
        for (int k = 0; k < 6; ++k) unpack16<PREC_F32>(__ldcs(xp + (size_t)k * x.vh), xv + 4 * k, 1.0f);
        r.load(j, rv);
#pragma unroll
        for (int k = 0; k < 24; ++k) {
            xv[k] = fmaf(al, pv[k], xv[k]);
            pv[k] = fmaf(be, pv[k], rv[k]);
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) __stcs(xp + (size_t)k * x.vh, pack16<PREC_F32>(xv + 4 * k, 1.0f));
        p.store(j, pv);
    }
    __device__ __forceinline__ void finish(const double (&)[1]) const {}
};

// x += x_lo + alpha p for the FP64 solution x, and x_lo = 0: the start of a
// reliable update, with the step of the last iteration (not yet in x_lo).  DFX: the
// new x in double-word form too, for the update's operator: that copy as a pass of
// its own reads x again and takes 29 us on 24^3 x 48, this whole one 59 us (820
// bytes per site, 4.6 TB/s).
template <int PX, int P, bool DFX> struct OpFlushX {
    static constexpr int NR = 0;
    FieldRef<PREC_F64> x;
    FieldRef<PX> xlo;
    FieldRef<P> p;
    FieldRef<PREC_DF> xd;
    const double *alpha;
    __device__ __forceinline__ void site(int j, double (&)[1]) const
    {
        using TX = typename Prec<PX>::real;
        const TX al = (TX)*alpha;
        TX lo[24];
        typename Prec<P>::real pv[24];
        xlo.load(j, lo);
        p.load(j, pv);
#pragma unroll
        for (int k = 0; k < 24; ++k) lo[k] = fma(al, to_real<TX>(pv[k]), lo[k]);
        const int h = j >= x.vh, i = j - h * x.vh;
#pragma unroll
        for (int k = 0; k < 12; ++k) {   // planes of two reals, the same in both formats
            const size_t o = h * x.half_bytes + ((size_t)k * x.vh + i) * 16;
            double v[2];
            unpack16<PREC_F64>(ldg16(x.p + o), v, 1.0f);
            v[0] += to_real<double>(lo[2 * k]);
            v[1] += to_real<double>(lo[2 * k + 1]);
            stg16(x.p + o, pack16<PREC_F64>(v, 1.0f));
            if constexpr (DFX) {
                const df d[2] = {to_real<df>(v[0]), to_real<df>(v[1])};
                stg16(xd.p + o, pack16<PREC_DF>(d, 1.0f));
            }
        }
#pragma unroll
        for (int k = 0; k < 24; ++k) lo[k] = TX(0);
        xlo.store(j, lo);
    }
    __device__ __forceinline__ void finish(const double (&)[1]) const {}
};

// y = a x + b y   (no reduction); UNIT (FP64 y): b = 1, one operation a real, chosen
// by the host: a test of b in the kernel is predicated and issues both forms'
// FP64 instructions on every element
template <int PX, int PY, bool UNIT = false> struct OpAxpby {
    static constexpr int NR = 0, FLAT = PX == PREC_F64 && PY == PREC_F64 ? 12 : 0;
    FieldRef<PX> x;
    FieldRef<PY> y;
    double a, b;
    struct In {
        uint4 x, y;
    };
    // vector k of both fields (half fields follow one another)
    __device__ __forceinline__ In vload(size_t k) const { return {ldg16(x.p + k * 16), ldg16(y.p + k * 16)}; }
    __device__ __forceinline__ void vuse(size_t k, const In &w) const
    {
        double xv[2], yv[2];
        unpack16<PREC_F64>(w.x, xv, 1.0f);
        unpack16<PREC_F64>(w.y, yv, 1.0f);
#pragma unroll
        for (int i = 0; i < 2; ++i) yv[i] = fma(a, xv[i], UNIT ? yv[i] : b * yv[i]);
        stg16(y.p + k * 16, pack16<PREC_F64>(yv, 1.0f));
    }
    __device__ __forceinline__ void site(int j, double (&)[1]) const
    {
        using T = typename Prec<PY>::real;
        typename Prec<PX>::real xv[24];
        T yv[24];
        x.load(j, xv);
        y.load(j, yv);
        const T ta = (T)a, tb = (T)b;
        if (PY == PREC_F64 ? UNIT : b == 1.0) {
#pragma unroll
            for (int k = 0; k < 24; ++k) yv[k] = fma(ta, to_real<T>(xv[k]), yv[k]);
        } else {
#pragma unroll
            for (int k = 0; k < 24; ++k) yv[k] = fma(ta, to_real<T>(xv[k]), tb * yv[k]);
        }
        y.store(j, yv);
    }
    __device__ __forceinline__ void finish(const double (&)[1]) const {}
};

// dst = src with a change of storage precision (no reduction)
template <int PD, int PS> struct OpConvert {
    static constexpr int NR = 0;
    FieldRef<PD> dst;
    FieldRef<PS> src;
    __device__ __forceinline__ void site(int j, double (&)[1]) const
    {
        typename Prec<PS>::real sv[24];
        typename Prec<PD>::real dv[24];
        src.load(j, sv);
#pragma unroll
        for (int k = 0; k < 24; ++k) dv[k] = to_real<typename Prec<PD>::real>(sv[k]);
        dst.store(j, dv);
    }
    __device__ __forceinline__ void finish(const double (&)[1]) const {}
};

} // namespace wd
