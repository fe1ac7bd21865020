// Vector updates and scalars of the streamed FP32 inner BiCGStab (bicg_f32.cu).  Every call takes
// `live`, a device word with the number of active right-hand sides: at zero its kernel returns at once.
#pragma once
#include "blas.cuh"

namespace laph {

// Partial sums of K complex values per right-hand side: item i, value k of right-hand side r at
//   f32: float2 p[(r >> 5) K kstride + i istride + k kstride + (r & 31)]   (stencil warps)
//   else c64 p[i istride + k kstride + r]
struct PartSums {
    const void *p;
    int count;
    long istride, kstride;
    bool f32;
};

// live = number of active right-hand sides
void bicg32_start(int nr, const BicgScalars &sc, int *live, cudaStream_t s);
// K = 1: <rhat, t>; K = 4: <t, s>, <t, t>, <rhat, t>, <rhat, s>
PartSums bicg32_dots(laph_ctx *ctx, long nrows, int nr, int K, const int *live, const cpx<float> *t, const cpx<float> *sv,
                     const uint32_t *code, cudaStream_t s);
// the convergence test on the residual of the last bicg32_xrp (not when first), then alpha (not when rv.p is null)
void bicg32_alpha(laph_ctx *ctx, long nrows, int nr, const BicgScalars &sc, bool first, const PartSums &rv, int *live,
                  cudaStream_t s);
// omega, rho and beta from the four products
void bicg32_omega(int nr, const BicgScalars &sc, const PartSums &ps, const int *live, cudaStream_t s);
// r <- r - alpha v
void bicg32_s(laph_ctx *ctx, long nrows, int nr, const BicgScalars &sc, const int *live, cpx<float> *r,
              const cpx<float> *v, cudaStream_t s);
// x += alpha p + omega s, r = s - omega t (s in r), p = r + beta (p - omega v)
void bicg32_xrp(laph_ctx *ctx, long nrows, int nr, const BicgScalars &sc, const int *live, cpx<float> *x, cpx<float> *r,
                cpx<float> *p, const cpx<float> *t, const cpx<float> *v, cudaStream_t s);

}  // namespace laph
