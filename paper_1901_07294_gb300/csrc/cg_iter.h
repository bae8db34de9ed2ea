// The four hops of one mixed-precision CG iteration with the vector work they
// carry (dslash_cg.cuh).
#pragma once

#include "wd_internal.h"

namespace wd {

struct CgFields {
    const char *p;            // search direction (even half field of the inner precision)
    char *r, *t_o, *t_e;      // residual (updated), scratch half fields
    float *site;              // one number per site (scratch)
    double *s;                // scalars: s[0] = |r|^2 in, s[1] = <p, A p>, s[2] = alpha, s[6] = breakdown flag out
    double *partials;         // reduction scratch
    unsigned *ticket;
};

// alpha = |r|^2 / |Mhat p|^2 and r -= alpha Mhat^dagger Mhat p, with each site's
// new |r|^2 in f.site; prec: FP32, FP16 or BF16.
int cg_iteration_hops(const wd_gauge *g, int prec, int recon, double mass, const CgFields &f, cudaStream_t s);

} // namespace wd
