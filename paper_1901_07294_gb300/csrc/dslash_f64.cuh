// FP64 hop with three threads per site.
//
// The FP64 hop is bound by the FP64 pipe (16 cycles per warp instruction and SM;
// 888 instructions per site), so on large lattices it needs enough warps to
// keep the pipe busy, and on small ones enough SMs.  As in dslash_df.cuh warp r of a
// 96-thread block computes colour row r of 32 consecutive sites and the block
// exchanges the projected half spinors through shared memory: a third of the
// per-site state, so 24 warps per SM without spills (one site per thread: 16
// warps, 200-550 bytes of spills), and three times the warps on a small lattice.
// The operations on a site and their order are those of hop_site's schedule 0.
// One site per thread against this kernel, even-odd hop: 24^3 x 48 with the axpy
// term 546 -> 522 us (467 at the pipe's rate), without 515 -> 507, 12^3 x 24 with it
// 61.8 -> 40.4, 16^4 without 58.5 -> 54.0, 8^4 31.6 -> 12.2 us; full operator on 32^4
// 1628 -> 1625 us.
// (Taking the two directions of a mu in one chain, s = U h + U^dagger h' for the
// upper spins and 2 U h - s for the lower ones, needs 840 instructions and 505 us on
// 24^3 x 48, but adds to the rounding error; not kept.)
#pragma once

#include "dslash_df.cuh"

namespace wd {

// resident blocks per SM the register budget is set for (80 registers; 12-real
// links, whose rebuilt row needs more: 136)
template <int RECON> constexpr int f64_row_blocks = RECON == 12 ? 5 : 8;

// [colour][h0, h1][site]; with 12-real links rec[c] holds entry (2, c) of the
// direction's link, rebuilt by warp c.
template <int RECON> struct F64HalfTile {
    double2 v[3][2][32];
    double2 rec[RECON == 12 ? 3 : 1][32];
};

// Entry (2, C) of a 12-real link (as Link::assemble).
template <int C>
__device__ __forceinline__ cpx<double> f64_row3_entry(const cpx<double> (&e0)[3], const cpx<double> (&e1)[3])
{
    constexpr int a = (C + 1) % 3, b = (C + 2) % 3;
    const cpx<double> x = e0[a], y = e1[b], z = e0[b], w = e1[a];
    double re = x.re * y.re;
    re = fma(-x.im, y.im, re);
    re = fma(-z.re, w.re, re);
    re = fma(z.im, w.im, re);
    double im = -(x.re * y.im);
    im = fma(-x.im, y.re, im);
    im = fma(z.re, w.im, im);
    im = fma(z.im, w.re, im);
    return {re, im};
}

// -v for m = 0x80000000, v for m = 0, off the FP64 pipe
__device__ __forceinline__ double flip_sign(double v, int m)
{
    return __hiloint2double(__double2hiint(v) ^ m, __double2loint(v));
}

// One direction for colour row r: acc += the colour-r components of
// (1 + S gamma_MU) U psi (FWD) or (1 + S gamma_MU) U^dagger psi.  neg: the sign of
// an antiperiodic boundary.  One barrier; the tile of a direction is rewritten two
// directions later, after the next barrier.
template <int MU, int S, bool FWD, int RECON, bool FIRST = false>
__device__ __forceinline__ void f64_row_dir(const char *in, const char *lblk, int vh, int nb, int li, bool neg, int r,
                                            int lane, F64HalfTile<RECON> &tile, cpx<double> (&acc)[4][1])
{
    cpx<double> p[4];
#pragma unroll
    for (int sp = 0; sp < 4; ++sp) {   // plane 3 sp + r holds (spin sp, colour r)
        double v[2];
        unpack16<PREC_F64>(ldg16(in + ((size_t)(3 * sp + r) * vh + nb) * 16), v, 1.0f);
        p[sp] = {v[0], v[1]};
    }
    cpx<double> u[3];   // U[r][c] (FWD) or U[c][r]
    auto entry = [&](int k) {   // plane k = 3 row + column holds one complex number
        double v[2];
        unpack16<PREC_F64>(ldg16(lblk + ((size_t)k * vh + li) * 16), v, 1.0f);
        return cpx<double>{v[0], v[1]};
    };
    if constexpr (RECON == 18) {
#pragma unroll
        for (int c = 0; c < 3; ++c) u[c] = entry(FWD ? 3 * r + c : 3 * c + r);
    } else {
        cpx<double> e0[3], e1[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            e0[c] = entry(c);
            e1[c] = entry(3 + c);
        }
        const cpx<double> rec = r == 0 ? f64_row3_entry<0>(e0, e1) : r == 1 ? f64_row3_entry<1>(e0, e1)
                                                                            : f64_row3_entry<2>(e0, e1);
        if constexpr (FWD) tile.rec[r][lane] = make_double2(rec.re, rec.im);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if constexpr (FWD) u[c] = r == 0 ? e0[c] : e1[c];   // row 2: from the tile below
            else u[c] = c == 2 ? rec : (r == 0 ? (c == 0 ? e0[0] : e1[0]) : r == 1 ? (c == 0 ? e0[1] : e1[1])
                                                                             : (c == 0 ? e0[2] : e1[2]));
        }
    }
    cpx<double> g0, g1;
    project_colour<MU, S>(p, g0, g1);
    if constexpr (MU == 3) {
        const int m = neg ? 0x80000000 : 0;
        g0 = {flip_sign(g0.re, m), flip_sign(g0.im, m)};
        g1 = {flip_sign(g1.re, m), flip_sign(g1.im, m)};
    }
    tile.v[r][0][lane] = make_double2(g0.re, g0.im);
    tile.v[r][1][lane] = make_double2(g1.re, g1.im);
    __syncthreads();
    if constexpr (RECON == 12 && FWD) {
        if (r == 2)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double2 q = tile.rec[c][lane];
                u[c] = {q.x, q.y};
            }
    }
    cpx<double> w0[1], w1[1];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double2 a = tile.v[c][0][lane], b = tile.v[c][1][lane];
        const cpx<double> h0{a.x, a.y}, h1{b.x, b.y};
        if (c == 0) {
            w0[0] = FWD ? cmul(u[c], h0) : cmul_conj(u[c], h0);
            w1[0] = FWD ? cmul(u[c], h1) : cmul_conj(u[c], h1);
        } else {
            w0[0] = FWD ? cfma(u[c], h0, w0[0]) : cfma_conj(u[c], h0, w0[0]);
            w1[0] = FWD ? cfma(u[c], h1, w1[0]) : cfma_conj(u[c], h1, w1[0]);
        }
    }
    accumulate<MU, S, FIRST>(acc, w0, w1);
}

// 18- or 12-real links; blocks alternate parity for the full operator as in
// hop_kernel; out = a x + b acc.  Threads past the last site compute the last
// site and store nothing: every thread takes part in the barriers.
template <int RECON, bool DAG, bool HAS_X>
__global__ void __launch_bounds__(DF_ROW_THREADS, f64_row_blocks<RECON>) hop_f64_row_kernel(const HopArgs A)
{
    grid_dependency_enter();
    __shared__ F64HalfTile<RECON> tile[2];
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
    cpx<double> acc[4][1];
    f64_row_dir<0, SF, true, RECON, true>(in, gf + 0 * lb, vh, nb[0], i, false, r, lane, tile[0], acc);
    f64_row_dir<0, SB, false, RECON>(in, gb + 0 * lb, vh, nb[4], nb[4], false, r, lane, tile[1], acc);
    f64_row_dir<1, SF, true, RECON>(in, gf + 1 * lb, vh, nb[1], i, false, r, lane, tile[0], acc);
    f64_row_dir<1, SB, false, RECON>(in, gb + 1 * lb, vh, nb[5], nb[5], false, r, lane, tile[1], acc);
    f64_row_dir<2, SF, true, RECON>(in, gf + 2 * lb, vh, nb[2], i, false, r, lane, tile[0], acc);
    f64_row_dir<2, SB, false, RECON>(in, gb + 2 * lb, vh, nb[6], nb[6], false, r, lane, tile[1], acc);
    f64_row_dir<3, SF, true, RECON>(in, gf + 3 * lb, vh, nb[3], i, ntf, r, lane, tile[0], acc);
    f64_row_dir<3, SB, false, RECON>(in, gb + 3 * lb, vh, nb[7], nb[7], ntb, r, lane, tile[1], acc);
    if (!active) return;

    const double a = A.a, b = A.b;
    char *out = (p ? A.out[1] : A.out[0]) + roff;
    const char *x = HAS_X ? (p ? A.x[1] : A.x[0]) + roff : nullptr;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const size_t off = ((size_t)(3 * s + r) * vh + i) * 16;   // plane of (spin s, colour r)
        double o[2] = {acc[s][0].re, acc[s][0].im};
        if constexpr (HAS_X) {
            double xv[2];
            unpack16<PREC_F64>(ldg16(x + off), xv, 1.0f);
            // b acc rounded, not a x: exact for the full operator's b = -1/2
            o[0] = fma(a, xv[0], b * o[0]);
            o[1] = fma(a, xv[1], b * o[1]);
        } else if (b != 1.0) {   // the bare hopping term needs no scaling
            o[0] *= b;
            o[1] *= b;
        }
        stg16(out + off, pack16<PREC_F64>(o, 1.0f));
    }
}

template <int RECON, bool DAG, bool HX>
cudaError_t launch_hop_f64_row(const HopArgs &A, int nrhs, cudaStream_t s)
{
    const int per = (A.vh + 31) / 32;
    const dim3 grid((unsigned)(per * A.nparity), (unsigned)nrhs);
    constexpr size_t fixed = sizeof(F64HalfTile<RECON>[2]);
    const size_t pad = spread_smem((long long)grid.x * grid.y, f64_row_blocks<RECON>, fixed, A.beside != 0);
    if (pad > 0) {
        static std::atomic<unsigned long long> allowed{0};
        const cudaError_t e = allow_smem(hop_f64_row_kernel<RECON, DAG, HX>, allowed, fixed);
        if (e != cudaSuccess) return e;
    }
    return wd_launch(hop_f64_row_kernel<RECON, DAG, HX>, grid, dim3(DF_ROW_THREADS), pad, s, A);
}

} // namespace wd
