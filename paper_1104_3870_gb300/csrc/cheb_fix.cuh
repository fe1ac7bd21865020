// Chebyshev chains of the slice Laplacian in two-limb fixed point (cheb_fix.cu).
#pragma once
#include <vector>

#include "common.cuh"

namespace laph {

// y = a (-Delta) x + b x per slice, the coefficients as limbs over 2^e
struct ChebMap {
    int4 *ab = nullptr;   // [nt]: limbs of a, limbs of b
    int *e = nullptr;     // [nt]
    std::vector<int4> hab;
    std::vector<int> he;
    bool ok = false;      // finite coefficients
    void set(laph_ctx *ctx, const char *name, const std::vector<double> &a, const std::vector<double> &b, cudaStream_t s);
};

struct ChebFix {
    laph_ctx *ctx = nullptr;
    Geom g;
    const int4 *u = nullptr;   // [t][k][9][V3] link limbs; null where the links are not bounded by one or memory is short
    longlong2 *f[3] = {};      // `chunk` vectors of every slice each, and their exponents
    short *e[3] = {};
    int chunk = 0;
    // builds the link limbs (synchronises); they stay null for links the format does not hold.  nvec: the most
    // vectors of a slice that a chain will get
    void init(laph_ctx *c, const Geom &geom, const c64 *U, int nvec, cudaStream_t s);
    bool usable(const ChebMap &m) const { return u && m.ok; }
    // out = T_order(map) in for nvec vectors of every slice; vector v of slice t at base + t * tstride + v * 3 V3
    void chain(const ChebMap &m, int order, int nvec, const c64 *in, long in_ts, c64 *out, long out_ts, cudaStream_t s) const;
};

}  // namespace laph
