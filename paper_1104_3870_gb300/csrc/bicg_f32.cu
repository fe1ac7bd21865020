// Vector updates and scalars of the streamed FP32 inner BiCGStab (the coded shadow vector of blas.cuh).
//
// With <rhat, r_new> = <rhat, s> - omega <rhat, t> from the stencil's epilogue, beta is known before the
// updates, so x, r and p are updated in one pass (read x, s, p, t, v, write x, r, p: 8 streams, where
// p = r + beta (p - omega v) on its own and x, r with their products took 10), and s overwrites r.
// An iteration is eight launches: two hops, alpha, s, two hops, omega, update; the sums over partial
// sums are done by the scalar kernels, one block per right-hand side.  The residual norm of an iteration
// is judged with the next alpha; once no right-hand side is active every kernel returns at once (*live
// == 0), so iterations queued past convergence cost launches only.
// 24^3 x 32, 32 right-hand sides (680 MB a stream): update 766 us (7.1 TB/s) and s 275 us, 1515 us an
// iteration with p, s and x, r in passes of their own and one right-hand side per thread.
#include "blas.cuh"
#include "bicg_f32.cuh"

namespace laph {

namespace {

__device__ __forceinline__ float2 f2mad(float2 a, float2 b, float2 c) {   // a b + c, complex
    return make_float2(fmaf(-a.y, b.y, fmaf(a.x, b.x, c.x)), fmaf(a.y, b.x, fmaf(a.x, b.y, c.y)));
}
template <int V>
struct Pack;
template <>
struct Pack<1> {
    using T = float2;
    static __device__ __forceinline__ float2 get(T v, int) { return v; }
    static __device__ __forceinline__ void set(T &v, int, float2 z) { v = z; }
};
template <>
struct Pack<2> {
    using T = float4;
    static __device__ __forceinline__ float2 get(T v, int k) { return k ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }
    static __device__ __forceinline__ void set(T &v, int k, float2 z) {
        if (k) {
            v.z = z.x;
            v.w = z.y;
        } else {
            v.x = z.x;
            v.y = z.y;
        }
    }
};
__device__ __forceinline__ float2 neg_f(c64 a) { return make_float2(-(float)a.re, -(float)a.im); }
__device__ __forceinline__ float2 pos_f(c64 a) { return make_float2((float)a.re, (float)a.im); }

// r <- r - alpha v; nrp = nr / V packs a row
template <int V>
__global__ void __launch_bounds__(256) s_kernel(long nrows, int nrp, int rpb, BicgScalars sc, const int *live,
                                                typename Pack<V>::T *__restrict__ r, const typename Pack<V>::T *__restrict__ v) {
    using P = Pack<V>;
    if (*live == 0) return;
    const int k = threadIdx.x % nrp, row0 = threadIdx.x / nrp;
    float2 al[V];
#pragma unroll
    for (int e = 0; e < V; ++e) al[e] = neg_f(sc.alpha[k * V + e]);
    const long step = (long)gridDim.x * rpb;
    auto one = [&](typename P::T a, typename P::T b) {
#pragma unroll
        for (int e = 0; e < V; ++e) P::set(a, e, f2mad(al[e], P::get(b, e), P::get(a, e)));
        return a;
    };
    long row = (long)blockIdx.x * rpb + row0;
    for (; row + 3 * step < nrows; row += 4 * step) {
        typename P::T a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            a[q] = r[(row + q * step) * nrp + k];
            b[q] = v[(row + q * step) * nrp + k];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) r[(row + q * step) * nrp + k] = one(a[q], b[q]);
    }
    for (; row < nrows; row += step) r[row * nrp + k] = one(r[row * nrp + k], v[row * nrp + k]);
}

// x += alpha p + omega s, r = s - omega t (s in r), p = r + beta (p - omega v), partial[block][rhs] = <r, r>
template <int V>
__global__ void __launch_bounds__(256) xrp_kernel(long nrows, int nrp, int rpb, BicgScalars sc, const int *live,
                                                  typename Pack<V>::T *__restrict__ x, typename Pack<V>::T *__restrict__ r,
                                                  typename Pack<V>::T *__restrict__ p, const typename Pack<V>::T *__restrict__ t,
                                                  const typename Pack<V>::T *__restrict__ v, double *__restrict__ partial) {
    using P = Pack<V>;
    using T = typename P::T;
    if (*live == 0) return;
    extern __shared__ double xsm[];
    const int tid = threadIdx.x, k = tid % nrp, row0 = tid / nrp;
    float2 al[V], om[V], nom[V], be[V];
    float acc[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
        al[e] = pos_f(sc.alpha[k * V + e]);
        om[e] = pos_f(sc.omega[k * V + e]);
        nom[e] = neg_f(sc.omega[k * V + e]);
        be[e] = pos_f(sc.beta[k * V + e]);
        acc[e] = 0.f;
    }
    auto one = [&](long i, T xv, T sv, T pv, T tv, T vv) {
        T xn, rn, pn;
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const float2 s = P::get(sv, e), q = P::get(pv, e);
            const float2 re = f2mad(nom[e], P::get(tv, e), s);
            P::set(xn, e, f2mad(om[e], s, f2mad(al[e], q, P::get(xv, e))));
            P::set(rn, e, re);
            P::set(pn, e, f2mad(be[e], f2mad(nom[e], P::get(vv, e), q), re));
            acc[e] = fmaf(re.x, re.x, fmaf(re.y, re.y, acc[e]));
        }
        x[i] = xn;
        r[i] = rn;
        p[i] = pn;
    };
    const long step = (long)gridDim.x * rpb;
    long row = (long)blockIdx.x * rpb + row0;
    for (; row + step < nrows; row += 2 * step) {
        const long i = row * nrp + k, j = (row + step) * nrp + k;
        const T x0 = x[i], s0 = r[i], p0 = p[i], t0 = t[i], v0 = v[i];
        const T x1 = x[j], s1 = r[j], p1 = p[j], t1 = t[j], v1 = v[j];
        one(i, x0, s0, p0, t0, v0);
        one(j, x1, s1, p1, t1, v1);
    }
    if (row < nrows) {
        const long i = row * nrp + k;
        one(i, x[i], r[i], p[i], t[i], v[i]);
    }
    const int bd = blockDim.x;
#pragma unroll
    for (int e = 0; e < V; ++e) xsm[e * bd + tid] = (double)acc[e];
    __syncthreads();
    for (int st = rpb / 2; st > 0; st >>= 1) {
        if (row0 < st)
#pragma unroll
            for (int e = 0; e < V; ++e) xsm[e * bd + tid] += xsm[e * bd + tid + st * nrp];
        __syncthreads();
    }
    const int nr = nrp * V;
    if (row0 == 0)
#pragma unroll
        for (int e = 0; e < V; ++e) partial[(long)blockIdx.x * nr + k * V + e] = xsm[e * bd + k];
}

// <t, s>, <t, t>, <rhat, t>, <rhat, s>: the generic form of the stencil's epilogue (K = 4), and <rhat, v>
// (K = 1, s unused); partial[block][K][nr]
template <int K>
__global__ void __launch_bounds__(256) dots_kernel(long nrows, int nr, int rpb, const int *live, const c32 *__restrict__ t,
                                                   const c32 *__restrict__ s, const uint32_t *__restrict__ code,
                                                   c64 *__restrict__ partial) {
    if (*live == 0) return;
    extern __shared__ c64 dsm[];
    const int tid = threadIdx.x, bd = blockDim.x, r = tid % nr, row0 = tid / nr;
    c32 acc[K];
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = c32{0.f, 0.f};
    for (long row = (long)blockIdx.x * rpb + row0; row < nrows; row += (long)gridDim.x * rpb) {
        const long i = row * nr + r;
        const uint32_t q = (code[(row / 12) * nr + r] >> (2 * (int)(row % 12))) & 3u;
        const c32 tv = t[i];
        if (K == 1) {
            acc[0] += rhat_conj_mul(q, tv);
        } else {
            const c32 sv = s[i];
            acc[0] += cmul_conj(tv, sv);
            acc[1].re += norm2(tv);
            acc[2] += rhat_conj_mul(q, tv);
            acc[3] += rhat_conj_mul(q, sv);
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) dsm[k * bd + tid] = cvt<double>(acc[k]);
    __syncthreads();
    for (int st = rpb / 2; st > 0; st >>= 1) {
        if (row0 < st)
#pragma unroll
            for (int k = 0; k < K; ++k) dsm[k * bd + tid] += dsm[k * bd + tid + st * nr];
        __syncthreads();
    }
    if (row0 == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) partial[((long)blockIdx.x * K + k) * nr + r] = dsm[k * bd + r];
}

// Sum over the partial sums of one right-hand side, fixed order, FP64 (all threads get it)
template <int K>
__device__ __forceinline__ void sum_parts(const PartSums &ps, int r, c64 out[K], double *sm) {
    double a[2 * K];
#pragma unroll
    for (int k = 0; k < 2 * K; ++k) a[k] = 0.0;
    const long off = ps.f32 ? (long)(r >> 5) * ps.kstride * K + (r & 31) : r;
    for (int i = threadIdx.x; i < ps.count; i += blockDim.x) {
        const long o = off + i * ps.istride;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (ps.f32) {
                const float2 z = ((const float2 *)ps.p)[o + k * ps.kstride];
                a[2 * k] += (double)z.x;
                a[2 * k + 1] += (double)z.y;
            } else {
                const c64 z = ((const c64 *)ps.p)[o + k * ps.kstride];
                a[2 * k] += z.re;
                a[2 * k + 1] += z.im;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 2 * K; ++k) {
        for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_xor_sync(0xffffffffu, a[k], o);
        if ((threadIdx.x & 31) == 0) sm[(threadIdx.x >> 5) * 2 * K + k] = a[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        out[k] = c64{0.0, 0.0};
        for (int w = 0; w < (int)blockDim.x / 32; ++w) {
            out[k].re += sm[w * 2 * K + 2 * k];
            out[k].im += sm[w * 2 * K + 2 * k + 1];
        }
    }
    __syncthreads();
}

__device__ __forceinline__ c64 quot(c64 a, c64 b) {
    const double d = norm2(b);
    return c64{(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__device__ __forceinline__ void stop_rhs(const BicgScalars &sc, int k, int status, int *live) {
    sc.active[k] = 0;
    sc.status[k] = status;
    sc.alpha[k] = sc.omega[k] = sc.beta[k] = c64{0.0, 0.0};
    atomicSub(live, 1);
}

// The residual norm of the iteration before (rr, skipped when first), then alpha = rho / <rhat, v> (skipped
// with rv.p null).  status 3 marks a right-hand side without a next direction: converged or broken down.
__global__ void __launch_bounds__(256) alpha_check_kernel(BicgScalars sc, const double *__restrict__ rr_part, int rr_count,
                                                          int nr, int first, PartSums rv, int *live) {
    __shared__ double sm[16];
    const int r = blockIdx.x;
    // not by *live: other blocks count it down meanwhile, and the warps of a block have to agree.  active[r] is
    // written by this block alone, behind a barrier.
    if (!sc.active[r]) return;
    double rr = 0.0;
    if (!first) {
        for (int i = threadIdx.x; i < rr_count; i += blockDim.x) rr += rr_part[(long)i * nr + r];
        for (int o = 16; o > 0; o >>= 1) rr += __shfl_xor_sync(0xffffffffu, rr, o);
        if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = rr;
        __syncthreads();
        rr = 0.0;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) rr += sm[w];
        __syncthreads();
    }
    c64 d[1];
    if (rv.p) sum_parts<1>(rv, r, d, sm);
    if (threadIdx.x != 0) return;
    if (!first) {
        sc.rr[r] = rr;
        const int s = sc.status[r];
        if (!isfinite(rr)) return stop_rhs(sc, r, 2, live);
        if (rr <= sc.rr_stop[r]) return stop_rhs(sc, r, 1, live);
        if (s == 3) return stop_rhs(sc, r, 2, live);
    }
    if (!rv.p) return;
    sc.iters[r] += 1;
    const double dn = norm2(d[0]);
    if (!(dn > 0.0) || !isfinite(dn) || dn < 1e-60 * sc.rr[r] * sc.rr[r]) return stop_rhs(sc, r, 2, live);
    sc.alpha[r] = quot(sc.rho[r], d[0]);
}

// omega = <t, s> / <t, t>, rho_new = <rhat, s> - omega <rhat, t>, beta = (rho_new / rho)(alpha / omega)
__global__ void __launch_bounds__(256) omega_beta_kernel(BicgScalars sc, PartSums ps, const int *live) {
    __shared__ double sm[64];
    if (*live == 0) return;
    const int r = blockIdx.x;
    c64 d[4];
    sum_parts<4>(ps, r, d, sm);
    if (threadIdx.x != 0 || !sc.active[r]) return;
    const double tt = d[1].re;
    c64 om{0.0, 0.0};
    if (tt > 0.0 && isfinite(tt)) om = c64{d[0].re / tt, d[0].im / tt};   // else s = 0: the half step solved the system
    const c64 rn = d[3] - om * d[2];
    sc.omega[r] = om;
    if (norm2(om) == 0.0 || norm2(rn) == 0.0 || !isfinite(rn.re) || !isfinite(rn.im)) {
        sc.beta[r] = c64{0.0, 0.0};
        sc.status[r] = 3;
        return;
    }
    sc.beta[r] = quot(rn, sc.rho[r]) * quot(sc.alpha[r], om);
    sc.rho[r] = rn;
}

__global__ void live_kernel(int nr, BicgScalars sc, int *live) {
    int n = 0;
    for (int k = 0; k < nr; ++k) n += sc.active[k] != 0;
    *live = n;
}

// threads of a block: nrp packs x rpb rows, up to 256
struct Plan {
    int V, nrp, rpb, block;
    unsigned grid;
};
Plan plan_of(laph_ctx *ctx, long nrows, int nr) {
    Plan p;
    p.V = nr % 2 == 0 ? 2 : 1;
    p.nrp = nr / p.V;
    p.rpb = 1;
    while (p.nrp * p.rpb * 2 <= 256) p.rpb *= 2;
    p.block = p.nrp * p.rpb;
    const long want = (nrows + p.rpb - 1) / p.rpb, cap = 8L * (ctx->sm_count > 0 ? ctx->sm_count : 152);
    p.grid = (unsigned)(want < cap ? want : cap);
    return p;
}

}  // namespace

void bicg32_start(int nr, const BicgScalars &sc, int *live, cudaStream_t s) {
    live_kernel<<<1, 1, 0, s>>>(nr, sc, live);
    LAPH_LAUNCH_CHECK();
}

PartSums bicg32_dots(laph_ctx *ctx, long nrows, int nr, int K, const int *live, const c32 *t, const c32 *sv,
                     const uint32_t *code, cudaStream_t s) {
    const RedPlan pl = red_plan(ctx, nrows, nr);
    c64 *partial = (c64 *)ws_get(ctx, "bicg32:part", sizeof(c64) * pl.grid * K * nr);
    const size_t shm = sizeof(c64) * K * pl.block;
    prof_begin("blas_fp32", s);
    if (K == 1)
        dots_kernel<1><<<pl.grid, pl.block, shm, s>>>(nrows, nr, pl.rpb, live, t, sv, code, partial);
    else
        dots_kernel<4><<<pl.grid, pl.block, shm, s>>>(nrows, nr, pl.rpb, live, t, sv, code, partial);
    LAPH_LAUNCH_CHECK();
    prof_end("blas_fp32", s, ((K == 1 ? 1.0 : 2.0) * sizeof(c32) + 4.0 / 12.0) * nrows * nr, 0.0);
    return PartSums{partial, (int)pl.grid, (long)K * nr, (long)nr, false};
}

void bicg32_alpha(laph_ctx *ctx, long nrows, int nr, const BicgScalars &sc, bool first, const PartSums &rv, int *live,
                  cudaStream_t s) {
    const Plan p = plan_of(ctx, nrows, nr);
    const double *rr = (const double *)ws_get(ctx, "bicg32:rr", sizeof(double) * p.grid * nr);
    alpha_check_kernel<<<nr, 256, 0, s>>>(sc, rr, (int)p.grid, nr, first ? 1 : 0, rv, live);
    LAPH_LAUNCH_CHECK();
}

void bicg32_omega(int nr, const BicgScalars &sc, const PartSums &ps, const int *live, cudaStream_t s) {
    omega_beta_kernel<<<nr, 256, 0, s>>>(sc, ps, live);
    LAPH_LAUNCH_CHECK();
}

void bicg32_s(laph_ctx *ctx, long nrows, int nr, const BicgScalars &sc, const int *live, c32 *r, const c32 *v, cudaStream_t s) {
    const Plan p = plan_of(ctx, nrows, nr);
    prof_begin("blas_fp32", s);
    if (p.V == 2)
        s_kernel<2><<<p.grid, p.block, 0, s>>>(nrows, p.nrp, p.rpb, sc, live, (float4 *)r, (const float4 *)v);
    else
        s_kernel<1><<<p.grid, p.block, 0, s>>>(nrows, p.nrp, p.rpb, sc, live, (float2 *)r, (const float2 *)v);
    LAPH_LAUNCH_CHECK();
    prof_end("blas_fp32", s, 3.0 * nrows * nr * sizeof(c32), 0.0);
}

void bicg32_xrp(laph_ctx *ctx, long nrows, int nr, const BicgScalars &sc, const int *live, c32 *x, c32 *r, c32 *p,
                const c32 *t, const c32 *v, cudaStream_t s) {
    const Plan pl = plan_of(ctx, nrows, nr);
    double *rr = (double *)ws_get(ctx, "bicg32:rr", sizeof(double) * pl.grid * nr);
    const size_t shm = sizeof(double) * pl.V * pl.block;
    prof_begin("blas_fp32", s);
    if (pl.V == 2)
        xrp_kernel<2><<<pl.grid, pl.block, shm, s>>>(nrows, pl.nrp, pl.rpb, sc, live, (float4 *)x, (float4 *)r, (float4 *)p,
                                                     (const float4 *)t, (const float4 *)v, rr);
    else
        xrp_kernel<1><<<pl.grid, pl.block, shm, s>>>(nrows, pl.nrp, pl.rpb, sc, live, (float2 *)x, (float2 *)r, (float2 *)p,
                                                     (const float2 *)t, (const float2 *)v, rr);
    LAPH_LAUNCH_CHECK();
    prof_end("blas_fp32", s, 8.0 * nrows * nr * sizeof(c32), 0.0);
}

}  // namespace laph
