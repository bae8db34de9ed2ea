// Double-word FP32 hop with three threads per site.
//
// The per-site kernel in double-word arithmetic needs about 250 registers a
// thread (a value is two FP32 registers, and its error terms add more), so only
// 8 warps fit on an SM, too few to hide the dependent chains of the error-free
// transformations.  Here warp r of a 96-thread block computes colour row r of
// the output for 32 consecutive checkerboard sites.  For each direction warp r
// loads the neighbours' colour-r spin components and projects them, the block
// exchanges the projected half spinors through shared memory, and each thread
// multiplies them by row r of U (column r for U^dagger) and accumulates the four
// spin components of colour r.  That is about a third of the per-site state,
// so more warps fit.  With 12-real links each warp also rebuilds one entry of
// the link's third row and shares it through the same tile.
//
// Two things bounded this form at 147 us on 24^3 x 48 (even-odd, axpy term; the
// bytes take 85 us): instruction issue, 70 % busy, and the wait for each
// direction's loads at its barrier.  The products and sums of the two spin
// components are now paired FP32 instructions, one issue slot for both (143 us),
// and the next direction's data is copied to shared memory meanwhile: 125 us.
// Full operator on 32^4 465 -> 364 us; 12-real links (paired only) 614 -> 562 us.
#pragma once

#include "dslash_impl.cuh"
#include "dslash_mrhs.cuh"
#include "dslash_pair.cuh"

namespace wd {

constexpr int DF_ROW_THREADS = 96;
// resident blocks per SM the register budget is set for.  18-real links: at most 97
// registers, of which the build takes 80, with 22.5 KB of shared memory, so that 8 blocks
// are resident; 12-real: 80, 9.2 KB, 124 bytes spilt.
template <int RECON> constexpr int df_row_blocks = RECON == 12 ? 8 : 7;

// (h0, h1) = upper two spin components of (1 + S gamma_MU) psi for one colour,
// from its four spin components p[s] (the table of project).
template <int MU, int S, typename T>
__device__ __forceinline__ void project_colour(const cpx<T> (&p)[4], cpx<T> &h0, cpx<T> &h1)
{
    if constexpr (MU == 0) {        // h0 = p0 + S i p3, h1 = p1 + S i p2
        h0 = {p[0].re - S * p[3].im, p[0].im + S * p[3].re};
        h1 = {p[1].re - S * p[2].im, p[1].im + S * p[2].re};
    } else if constexpr (MU == 1) { // h0 = p0 - S p3, h1 = p1 + S p2
        h0 = {p[0].re - S * p[3].re, p[0].im - S * p[3].im};
        h1 = {p[1].re + S * p[2].re, p[1].im + S * p[2].im};
    } else if constexpr (MU == 2) { // h0 = p0 + S i p2, h1 = p1 - S i p3
        h0 = {p[0].re - S * p[2].im, p[0].im + S * p[2].re};
        h1 = {p[1].re + S * p[3].im, p[1].im - S * p[3].re};
    } else {                        // h0 = p0 + S p2, h1 = p1 + S p3
        h0 = {p[0].re + S * p[2].re, p[0].im + S * p[2].im};
        h1 = {p[1].re + S * p[3].re, p[1].im + S * p[3].im};
    }
}

// ---- pairs of double-word numbers -------------------------------------------
// The two spin components that the projected form carries through a direction
// run through the same operations, so they are held as pairs (lanes x and y)
// and computed with Blackwell's paired FP32 instructions: one issue slot for
// both.  The kernel is bound by instruction issue (70 % active before, 10,930
// instructions per site), not by the FMA pipe (60 %).
struct dfp {
    f2 hi, lo;
};

__device__ __forceinline__ f2 q_sub(f2 a, f2 b)
{
    f2 r;
    asm("{.reg .b64 a, b, c; mov.b64 a, {%2, %3}; mov.b64 b, {%4, %5}; sub.rn.f32x2 c, a, b; mov.b64 {%0, %1}, c;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// a += (SX, SY) x lane-wise (+1 or -1) without renormalising: the running sum
// of a compensated dot product, normalised once before it is used as a product
// operand (a lo part that grew past hi would lose accuracy there).  The signs
// ride on FMAs, whose products are exact.
template <int SX, int SY> __device__ __forceinline__ void lazy_acc(dfp &a, const dfp &x)
{
    const f2 g = make_float2((float)SX, (float)SY);
    constexpr bool plus = SX > 0 && SY > 0;
    const f2 s = plus ? p_add(a.hi, x.hi) : p_fma(g, x.hi, a.hi);
    const f2 nb = q_sub(a.hi, s);               // -(s - a)
    const f2 t1 = q_sub(a.hi, p_add(s, nb));
    const f2 t2 = plus ? p_add(x.hi, nb) : p_fma(g, x.hi, nb);
    const f2 l = plus ? p_add(a.lo, x.lo) : p_fma(g, x.lo, a.lo);
    a = {s, p_add(p_add(t1, t2), l)};
}

// One real part of a link entry in both lanes, with its negative.
struct dfu {
    f2 h, l, nh, nl;
    __device__ __forceinline__ explicit dfu(df v)
        : h(p_bcast(v.hi)), l(p_bcast(v.lo)), nh(p_bcast(-v.hi)), nl(p_bcast(-v.lo))
    {
    }
};

// x y in both lanes as an FMA with zero: the compiler contracts a paired product
// and a following paired sum into one FMA, rounding once where the error terms
// need the rounded product
__device__ __forceinline__ f2 q_mul(f2 a, f2 b) { return p_fma(a, b, make_float2(0.0f, 0.0f)); }

// x y, not normalised: the product and its error terms
__device__ __forceinline__ dfp dfp_mul(const f2 h, const f2 l, const f2 nh, const dfp &y)
{
    const f2 np = q_mul(nh, y.hi);
    f2 e = p_fma(h, y.hi, np);
    e = p_fma(h, y.lo, e);
    e = p_fma(l, y.hi, e);
    return {q_mul(h, y.hi), e};
}

// z + x y, one compensated dot-product step (fma(df, df, df) in both lanes),
// with the product held negated so that no operand needs a sign of its own
__device__ __forceinline__ dfp dfp_fma(const f2 h, const f2 l, const f2 nh, const dfp &y, const dfp &z)
{
    const f2 np = q_mul(nh, y.hi);
    f2 e = p_fma(h, y.hi, np);
    e = p_fma(h, y.lo, e);
    e = p_fma(l, y.hi, e);
    const f2 s = q_sub(z.hi, np);
    const f2 b = q_sub(s, z.hi);
    const f2 t = q_sub(q_sub(z.hi, q_sub(s, b)), p_add(np, b));
    return {s, p_add(t, p_add(e, z.lo))};
}

// Accumulators of one colour row: the upper spins and, as in the spin-paired
// 16-bit kernel, the lower ones in the order the projector pairs them with
// (w0, w1): crosswise for x and y, straight for z and t.
struct DfAcc {
    dfp up_re, up_im;     // (acc_0, acc_1)
    dfp l32_re, l32_im;   // (acc_3, acc_2), from the x and y directions
    dfp l23_re, l23_im;   // (acc_2, acc_3), from the z and t directions
};

// accumulate for colour row r only, with lazy sums; FIRST: the first direction
// (MU = 0) assigns the upper and x, y sums, and the first of z, t (MU = 2) its own
template <int SX, int SY, bool SET> __device__ __forceinline__ void lazy_put(dfp &a, const dfp &x)
{
    if constexpr (SET) {
        const f2 g = make_float2((float)SX, (float)SY);
        a = SX > 0 && SY > 0 ? x : dfp{p_mul(g, x.hi), p_mul(g, x.lo)};
    } else lazy_acc<SX, SY>(a, x);
}
template <int MU, int S, bool FIRST>
__device__ __forceinline__ void df_accumulate(DfAcc &a, const dfp &wr, const dfp &wi)
{
    lazy_put<1, 1, FIRST && MU == 0>(a.up_re, wr);
    lazy_put<1, 1, FIRST && MU == 0>(a.up_im, wi);
    if constexpr (MU == 0) {        // spin3 += -S i w0, spin2 += -S i w1
        lazy_put<S, S, FIRST>(a.l32_re, wi);
        lazy_put<-S, -S, FIRST>(a.l32_im, wr);
    } else if constexpr (MU == 1) { // spin3 += -S w0, spin2 += S w1
        lazy_put<-S, S, FIRST>(a.l32_re, wr);
        lazy_put<-S, S, FIRST>(a.l32_im, wi);
    } else if constexpr (MU == 2) { // spin2 += -S i w0, spin3 += S i w1
        lazy_put<S, -S, FIRST>(a.l23_re, wi);
        lazy_put<-S, S, FIRST>(a.l23_im, wr);
    } else {                        // spin2 += S w0, spin3 += S w1
        lazy_put<S, S, FIRST>(a.l23_re, wr);
        lazy_put<S, S, FIRST>(a.l23_im, wi);
    }
}

// The projected half spinors of the block's 32 sites for one direction:
// warp c writes colour c, every warp then reads all three.  [colour][real or
// imaginary part][site], each as (h0.hi, h1.hi, h0.lo, h1.lo): two aligned
// pairs per load.  With 12-real links, rec[c] holds entry (2, c) of the
// direction's link, rebuilt by warp c.
template <int RECON> struct DfHalfTile {
    float4 v[3][2][32];
    float4 rec[RECON == 12 ? 3 : 1][32];
};

// Each thread's staging slots (18-real links): the next direction's neighbour
// components and link entries, brought in by asynchronous copies while this
// direction's products run; the entries double-buffered, being in use till then.
struct DfStage {
    uint4 p[4][DF_ROW_THREADS];
    uint4 u[2][3][DF_ROW_THREADS];
};

template <bool FWD>
__device__ __forceinline__ void df_stage(const char *in, const char *lblk, int vh, int nb, int li, int r, int buf,
                                         DfStage &st)
{
    const int tid = threadIdx.x;
#pragma unroll
    for (int sp = 0; sp < 4; ++sp)   // plane 3 sp + r holds (spin sp, colour r)
        copy_async<16>((unsigned)__cvta_generic_to_shared(&st.p[sp][tid]), in + ((size_t)(3 * sp + r) * vh + nb) * 16);
#pragma unroll
    for (int c = 0; c < 3; ++c)      // plane k = 3 row + column holds one complex number
        copy_async<16, true>((unsigned)__cvta_generic_to_shared(&st.u[buf][c][tid]),
                             lblk + ((size_t)(FWD ? 3 * r + c : 3 * c + r) * vh + li) * 16);
    copy_commit();
}

// Entry (2, C) of a 12-real link from its stored rows 0 and 1:
// conj(U0a U1b - U0b U1a) with a = C+1, b = C+2 (mod 3), one four-term
// compensated chain per part as in Link::load, normalised for use as a
// product operand.
template <int C>
__device__ __forceinline__ cpx<df> df_row3_entry(const cpx<df> (&e0)[3], const cpx<df> (&e1)[3])
{
    constexpr int a = (C + 1) % 3, b = (C + 2) % 3;
    const cpx<df> x = e0[a], y = e1[b], z = e0[b], w = e1[a];
    df re = x.re * y.re;
    re = fma(-x.im, y.im, re);
    re = fma(-z.re, w.re, re);
    re = fma(z.im, w.im, re);
    df im = -(x.re * y.im);
    im = fma(-x.im, y.re, im);
    im = fma(z.re, w.im, im);
    im = fma(z.im, w.re, im);
    return {df_normalize(re), df_normalize(im)};
}

// One direction for colour row r: acc += the colour-r components of
// (1 + S gamma_MU) U psi (FWD) or (1 + S gamma_MU) U^dagger psi.  Warp r takes
// the neighbour's colour-r spin components only and projects them (neg: with
// the sign of an antiperiodic boundary); the block exchanges the projections
// through `tile` (one barrier; the tile of a direction is rewritten two
// directions later, after the next barrier).
// 18-real links: components and entries come from this thread's slots of
// `stage`, filled a direction ahead; next() starts the copies for the next one.
// 12-real links: every warp loads the two stored rows and rebuilds entry
// (2, r); a forward hop's row 2 is then the three warps' entries, read from
// the tile after the same barrier.  (Staging their six entries costs the
// shared memory of two resident blocks: 32^4 full operator 649 us against 562.)
template <int MU, int S, bool FWD, int RECON, bool FIRST, typename Next>
__device__ __forceinline__ void df_row_dir(const char *in, const char *lblk, int vh, int nb, int li, bool neg, int r,
                                           int lane, DfHalfTile<RECON> &tile, DfStage &stage, int buf, DfAcc &acc,
                                           Next &&next)
{
    const int tid = threadIdx.x;
    cpx<df> p[4], u[3];   // u = U[r][c] (FWD) or U[c][r]
    auto number = [](uint4 w) {
        df v[2];
        unpack16<PREC_DF>(w, v, 1.0f);
        return cpx<df>{v[0], v[1]};
    };
    if constexpr (RECON == 18) {
        copy_wait<0>();
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) p[sp] = number(stage.p[sp][tid]);
    } else {
#pragma unroll
        for (int sp = 0; sp < 4; ++sp) p[sp] = number(ldg16(in + ((size_t)(3 * sp + r) * vh + nb) * 16));
        cpx<df> e0[3], e1[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            e0[c] = number(ldg16(lblk + ((size_t)c * vh + li) * 16));
            e1[c] = number(ldg16(lblk + ((size_t)(3 + c) * vh + li) * 16));
        }
        const cpx<df> rec = r == 0 ? df_row3_entry<0>(e0, e1) : r == 1 ? df_row3_entry<1>(e0, e1)
                                                                       : df_row3_entry<2>(e0, e1);
        tile.rec[r][lane] = make_float4(rec.re.hi, rec.re.lo, rec.im.hi, rec.im.lo);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if constexpr (FWD) u[c] = r == 0 ? e0[c] : e1[c];   // row 2: from the tile below
            else u[c] = c == 2 ? rec : (r == 0 ? (c == 0 ? e0[0] : e1[0]) : r == 1 ? (c == 0 ? e0[1] : e1[1])
                                                                             : (c == 0 ? e0[2] : e1[2]));
        }
    }
    cpx<df> g0, g1;
    project_colour<MU, S>(p, g0, g1);
    if (neg) {
        g0 = {-g0.re, -g0.im};
        g1 = {-g1.re, -g1.im};
    }
    tile.v[r][0][lane] = make_float4(g0.re.hi, g1.re.hi, g0.re.lo, g1.re.lo);
    tile.v[r][1][lane] = make_float4(g0.im.hi, g1.im.hi, g0.im.lo, g1.im.lo);
    next();   // refills the neighbour's slots, which this thread has read
    __syncthreads();
    if constexpr (RECON == 18) {
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = number(stage.u[buf][c][tid]);
    }
    if constexpr (RECON == 12 && FWD) {
        if (r == 2)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float4 q = tile.rec[c][lane];
                u[c] = {df(q.x, q.y), df(q.z, q.w)};
            }
    }
    dfp wr, wi;   // (w0, w1) = the colour-r component of U h or U^dagger h
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float4 a = tile.v[c][0][lane], b = tile.v[c][1][lane];
        const dfp hr{make_float2(a.x, a.y), make_float2(a.z, a.w)}, hi{make_float2(b.x, b.y), make_float2(b.z, b.w)};
        const dfu x(u[c].re), y(FWD ? u[c].im : -u[c].im);
        if (c == 0) {
            wr = dfp_mul(x.h, x.l, x.nh, hr);
            wi = dfp_mul(x.h, x.l, x.nh, hi);
        } else {
            wr = dfp_fma(x.h, x.l, x.nh, hr, wr);
            wi = dfp_fma(x.h, x.l, x.nh, hi, wi);
        }
        wr = dfp_fma(y.nh, y.nl, y.h, hi, wr);
        wi = dfp_fma(y.h, y.l, y.nh, hr, wi);
    }
    df_accumulate<MU, S, FIRST>(acc, wr, wi);
}

// 18- or 12-real links; blocks alternate parity for the full operator as in
// hop_kernel; out = a x + b acc.  Every thread of a block takes part in the
// barriers: threads past the last site compute the last site and store nothing.
template <int RECON, bool DAG, bool HAS_X>
__global__ void __launch_bounds__(DF_ROW_THREADS, df_row_blocks<RECON>) hop_df_row_kernel(const HopArgs A)
{
    grid_dependency_enter();
    __shared__ DfHalfTile<RECON> tile[2];
    __shared__ DfStage stage;   // unused (and not allocated) with 12-real links
    int p, blk;
    if (A.nparity == 2) { p = blockIdx.x & 1; blk = blockIdx.x >> 1; }
    else { p = A.parity0; blk = blockIdx.x; }
    const int r = threadIdx.x >> 5;   // warp-uniform
    const int lane = threadIdx.x & 31;
    const int vh = A.vh;
    const int i0 = blk * 32 + lane;
    const bool active = i0 < vh;
    const int i = active ? i0 : vh - 1;
    const size_t roff = (size_t)blockIdx.y * A.rhs_stride, lb = A.link_blk;
    const char *in = (p ? A.in[1] : A.in[0]) + roff;
    const char *gf = p ? A.gauge[1] : A.gauge[0];
    const char *gb = p ? A.gauge[0] : A.gauge[1];
    int nb[8];
    site_neighbours(A, p, i, nb);
    // a t hop wraps exactly when the neighbour's index falls below (forward) or above (backward) i
    const bool ntf = A.tneg && nb[3] < i, ntb = A.tneg && nb[7] > i;
    constexpr int SF = DAG ? +1 : -1;
    constexpr int SB = -SF;
    DfAcc acc;
    // directions x-, y-, z-, t-, x+, y+, z+, t+; the slots of direction k + 1 are
    // filled during direction k
    auto fill = [&](auto kc) {
        constexpr int k = decltype(kc)::value, mu = k & 3;
        if constexpr (RECON == 18 && k < 8) {
            if constexpr (k < 4) df_stage<false>(in, gb + mu * lb, vh, nb[4 + mu], nb[4 + mu], r, k & 1, stage);
            else df_stage<true>(in, gf + mu * lb, vh, nb[mu], i, r, k & 1, stage);
        }
    };
    auto hop = [&](auto kc) {
        constexpr int k = decltype(kc)::value, mu = k & 3;
        constexpr bool fwd = k >= 4, first = k == 0 || k == 2;
        df_row_dir<mu, fwd ? SF : SB, fwd, RECON, first>(in, (fwd ? gf : gb) + mu * lb, vh, nb[fwd ? mu : 4 + mu],
                                                         fwd ? i : nb[4 + mu], mu == 3 && (fwd ? ntf : ntb), r, lane,
                                                         tile[k & 1], stage, k & 1, acc,
                                                         [&] { fill(std::integral_constant<int, k + 1>{}); });
    };
    fill(std::integral_constant<int, 0>{});
    hop(std::integral_constant<int, 0>{});
    hop(std::integral_constant<int, 1>{});
    hop(std::integral_constant<int, 2>{});
    hop(std::integral_constant<int, 3>{});
    hop(std::integral_constant<int, 4>{});
    hop(std::integral_constant<int, 5>{});
    hop(std::integral_constant<int, 6>{});
    hop(std::integral_constant<int, 7>{});
    if (!active) return;

    // the four spins: 0, 1 from the upper pair, 2 and 3 from both lower pairs
    auto sum = [](float ah, float al, float bh, float bl) {
        const df t = df_two_sum(ah, bh);
        return df{t.hi, __fadd_rn(t.lo, __fadd_rn(al, bl))};
    };
    const cpx<df> spin[4] = {
        {df(acc.up_re.hi.x, acc.up_re.lo.x), df(acc.up_im.hi.x, acc.up_im.lo.x)},
        {df(acc.up_re.hi.y, acc.up_re.lo.y), df(acc.up_im.hi.y, acc.up_im.lo.y)},
        {sum(acc.l23_re.hi.x, acc.l23_re.lo.x, acc.l32_re.hi.y, acc.l32_re.lo.y),
         sum(acc.l23_im.hi.x, acc.l23_im.lo.x, acc.l32_im.hi.y, acc.l32_im.lo.y)},
        {sum(acc.l23_re.hi.y, acc.l23_re.lo.y, acc.l32_re.hi.x, acc.l32_re.lo.x),
         sum(acc.l23_im.hi.y, acc.l23_im.lo.y, acc.l32_im.hi.x, acc.l32_im.lo.x)}};
    const df a = (df)A.a, b = (df)A.b;
    char *out = (p ? A.out[1] : A.out[0]) + roff;
    const char *x = HAS_X ? (p ? A.x[1] : A.x[0]) + roff : nullptr;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const size_t off = ((size_t)(3 * s + r) * vh + i) * 16;   // plane of (spin s, colour r)
        const cpx<df> v = {df_normalize(spin[s].re), df_normalize(spin[s].im)};
        df o[2];
        if constexpr (HAS_X) {
            df xv[2];
            unpack16<PREC_DF>(ldg16(x + off), xv, 1.0f);
            o[0] = a * xv[0] + b * v.re;
            o[1] = a * xv[1] + b * v.im;
        } else if (A.b == 1.0) {
            o[0] = v.re;
            o[1] = v.im;
        } else {
            o[0] = b * v.re;
            o[1] = b * v.im;
        }
        stg16(out + off, pack16<PREC_DF>(o, 1.0f));
    }
}

template <int RECON, bool DAG, bool HX>
cudaError_t launch_hop_df_row(const HopArgs &A, int nrhs, cudaStream_t s)
{
    const int per = (A.vh + 31) / 32;
    return wd_launch(hop_df_row_kernel<RECON, DAG, HX>, dim3((unsigned)(per * A.nparity), (unsigned)nrhs),
                     dim3(DF_ROW_THREADS), 0, s, A);
}

} // namespace wd
