// The CG iteration's share of the hops.
//
// A = Mhat^dagger Mhat, so the step length needs no product with A p:
//     <p, A p> = |Mhat p|^2,
// known after the second of the iteration's four hops.  The hops therefore
// carry the iteration's vector work with them:
//   CG_NORM    second hop: out = Mhat p, and each site's |out|^2 (in the field's
//              compute type, 4 bytes a site) to a scratch array;
//   CG_ALPHA   third hop: its first CG_PARTS blocks add that array in FP64
//              and set alpha = |r|^2 / |Mhat p|^2, beside the blocks of the hop;
//   CG_RESID   fourth hop: A p stays in registers, r -= alpha A p is stored and
//              each site's |r|^2 goes to the scratch array.
// Left for kernels of their own are the sum of |r|^2 and the update of x and p
// (OpXp).  Compared with separate BLAS kernels for p = r + beta p, <p, A p>
// and the update of x and r, A p is neither written nor read again and p is
// read once instead of three times, in 6 launches instead of 8 (with the loop's
// control).  24^3 x 48, FP16 storage: 136 -> 120 us of kernel time an iteration
// (four hops 97 -> 99, the rest 39 -> 21); solves to 1e-12: FP16 21.6 -> 20.6 ms,
// FP32 32.5 -> 30.0 ms, 32^4 FP32 48.3 -> 43.7 ms, 16^4 FP16 4.9 -> 4.6 ms.
#pragma once

#include "blas.cuh"
#include "dslash_pair.cuh"

namespace wd {

enum { CG_NORM = 1, CG_ALPHA = 2, CG_RESID = 3 };

// Blocks that add one solve's site sums, fixed by the number of sites only (the
// order of the sum, and so its bits, must not depend on what else runs).
constexpr int CG_PARTS = 128;
__host__ __device__ __forceinline__ int cg_parts(int n, int threads)
{
    const int want = (n / 4 + 4 * threads - 1) / (4 * threads);   // about four loads a thread at least
    return want < CG_PARTS ? (want > 0 ? want : 1) : CG_PARTS;
}

// What the hops need of a solve: the residual, the site sums and the scalars
// (s[0] = |r|^2, s[1] = <p, A p>, s[2] = alpha, s[6] = breakdown flag).
struct CgHop {
    char *r;
    float *site;
    double *s;
    RedScratch red;
};

// Part `part` of `nparts` of the sum of site[0 .. n) in FP64, n a multiple of 4.
// The block that ends last adds the parts and calls finish(sum) in one thread,
// which is where true is returned.  At most 256 threads, in whole warps along x.
template <typename Finish>
__device__ __forceinline__ bool site_sum(const float *site, int n, int part, int nparts, const RedScratch &red,
                                         Finish &&finish)
{
    __shared__ double warp_sum[8];
    __shared__ bool last;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, nthr = blockDim.x * blockDim.y;
    const int lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
    // four running sums: a FP64 addition's latency is several times its issue time
    double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
    const float4 *q = reinterpret_cast<const float4 *>(site);
#pragma unroll 4
    for (int k = part * nthr + tid; k < n / 4; k += nparts * nthr) {
        const float4 w = __ldcg(q + k);
        v0 += f32_to_f64(w.x);
        v1 += f32_to_f64(w.y);
        v2 += f32_to_f64(w.z);
        v3 += f32_to_f64(w.w);
    }
    double v = (v0 + v1) + (v2 + v3);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) warp_sum[warp] = v;
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < nwarp; ++w) v += warp_sum[w];
        red.partials[part] = v;
        last = ticket_take(red.ticket) == (unsigned)nparts - 1u;
    }
    __syncthreads();
    if (!last || warp != 0) return false;
    v = 0.0;
#pragma unroll
    for (int k = 0; k < CG_PARTS / 32; ++k) v += 32 * k + lane < nparts ? __ldcg(red.partials + 32 * k + lane) : 0.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane != 0) return false;
    *red.ticket = 0u;   // ready for the next sum
    finish(v);
    return true;
}

// alpha = |r|^2 / <p, A p> (0 and the flag set on breakdown)
__device__ __forceinline__ void cg_set_alpha(double *s, double pap)
{
    s[1] = pap;
    const bool ok = pap > 0.0 && pap < 1e300;
    s[2] = ok ? s[0] / pap : 0.0;
    if (!ok) s[6] = 1.0;
}

// |v|^2 of a site in the order of OpNorm2
__device__ __forceinline__ float site_norm2(const float (&v)[24])
{
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 24; ++k) s = fmaf(v[k], v[k], s);
    return s;
}

// r -= alpha o at site i; its |r|^2
template <int P> __device__ __forceinline__ float cg_residual(char *r, int vh, int i, float alpha, const float (&o)[24])
{
    float v[24];
    Spinor<P>::load(r, vh, i, v);
#pragma unroll
    for (int k = 0; k < 24; ++k) v[k] = fmaf(-alpha, o[k], v[k]);
    Spinor<P>::store(r, vh, i, v);
    return site_norm2(v);
}

// The axpy terms (p in the second hop, Mhat p in the fourth) are read with the
// streaming hint: nothing needs them before the links have passed through L2 again
// (FP16 24^3 x 48 19.29 -> 19.20 ms a solve, FP32 28.56 -> 28.23, 32^4 41.47 ->
// 41.22).
template <int P> struct CgNormStore {
    float *site;
    __device__ __forceinline__ void operator()(const HopArgs &A, int p, int i, size_t roff,
                                               const cpx<float> (&acc)[4][3]) const
    {
        float o[24];
        hop_value<P, true, true>(A, p, i, roff, acc, o);
        site[i] = site_norm2(o);
        Spinor<P>::store((p ? A.out[1] : A.out[0]) + roff, A.vh, i, o);
    }
};

template <int P> struct CgResidStore {
    char *r;
    float *site;
    float alpha;
    __device__ __forceinline__ void operator()(const HopArgs &A, int p, int i, size_t roff,
                                               const cpx<float> (&acc)[4][3]) const
    {
        float o[24];
        hop_value<P, true, true>(A, p, i, roff, acc, o);
        site[i] = cg_residual<P>(r, A.vh, i, alpha, o);
    }
};

// One hop of the iteration with its share of the vector work, in memory schedule PF (0
// or 1) with or without L1 allocation for the links (LNA), as hop_kernel; 16-bit storage:
// the spin-paired kernel.
template <int P, int RECON, int STEP, int PF, bool LNA>
__global__ void __launch_bounds__(256, 2) hop_cg_kernel(const HopArgs A, const CgHop C, const int nparts)
{
    grid_dependency_enter();
    int blk = blockIdx.x;
    if constexpr (STEP == CG_ALPHA) {
        if (blk < nparts) {
            site_sum(C.site, A.vh, blk, nparts, C.red, [&](double v) { cg_set_alpha(C.s, v); });
            return;
        }
        blk -= nparts;
    }
    // every second hop runs through the lattice backwards: it starts on the links
    // and fields that the hop before it left in L2 (FP32, 24^3 x 48: 31.6 -> 30.3
    // ms a solve, FP16 on 32^4 32.8 -> 31.8; what a 16^4 solve touches fits in L2 anyway)
    if constexpr (STEP != CG_ALPHA) blk = gridDim.x - 1 - blk;
    const int i = blk * blockDim.x + threadIdx.x;
    if (i >= A.vh) return;
    constexpr bool DAG = STEP != CG_NORM, HX = STEP != CG_ALPHA;
    auto run = [&](const auto &epi) {
        if constexpr (Prec<P>::scaled) sp_site<P, RECON, DAG, HX, PF, LNA>(A, A.parity0, i, 0, epi);
        else hop_site<P, RECON, DAG, HX, PF, false, LNA>(A, A.parity0, i, 0, epi);
    };
    if constexpr (STEP == CG_NORM) run(CgNormStore<P>{C.site});
    else if constexpr (STEP == CG_ALPHA) run(HopStore<P, false>{});
    else run(CgResidStore<P>{C.r, C.site, (float)C.s[2]});
}

} // namespace wd
