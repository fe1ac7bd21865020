// The FP32 inner BiCGStab of a small lattice in one kernel: one thread-block cluster per right-hand
// side, from the first residual to convergence.
//
// On small lattices an iteration of the streamed solver (solver.cu) is ten to fourteen launches of a
// few microseconds each with almost nothing in them: 47 us an iteration on 4^3 x 8 with 8 right-hand
// sides.  Here four lanes own a site: lane mu takes the forward and backward hop of direction mu, the
// four partial sums are exchanged by shuffles, and lane mu forms the three components of spin mu.  A
// lane keeps its components of x, r, p, v, s and t in registers; only the operand of the next hop leaves
// it, through the shared memory of its CTA, which the cluster reads, between cluster barriers (six an
// iteration).  Inner products are FP32 products in two-float sums (48 bits), over lanes, warps and CTAs in
// a fixed order, so every CTA of a cluster takes the same decision; their error is the rounding of the
// products, 2^-24 as in the streamed solver.
//
// The recurrences are those of solver.cu with the coded shadow vector of blas.cuh, with two changes
// that save a barrier: <rhat, r> of the new residual is <rhat, s> - omega <rhat, t>, and <r, r> is summed
// with the next <rhat, v>, so convergence is seen half an iteration later.
#include <cooperative_groups.h>

#include "blas.cuh"
#include "dirac.cuh"
#include "solver.cuh"

namespace laph {

namespace cg = cooperative_groups;

namespace {

constexpr int SB_NRED = 8;     // reals of one reduction

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 ci(float2 a) { return make_float2(-a.y, a.x); }
// a + b c, a + conj(b) c
__device__ __forceinline__ float2 cfma(float2 b, float2 c, float2 a) {
    return make_float2(fmaf(-b.y, c.y, fmaf(b.x, c.x, a.x)), fmaf(b.y, c.x, fmaf(b.x, c.y, a.y)));
}
__device__ __forceinline__ float2 cfma_conj(float2 b, float2 c, float2 a) {
    return make_float2(fmaf(b.y, c.y, fmaf(b.x, c.x, a.x)), fmaf(-b.y, c.x, fmaf(b.x, c.y, a.y)));
}

// two-float sums
struct F2 {
    float h, l;
};
__device__ __forceinline__ F2 two_add(F2 a, F2 b) {
    const float s = a.h + b.h, bb = s - a.h;
    const float e = (a.h - (s - bb)) + (b.h - bb) + (a.l + b.l);
    const float h = s + e;
    return {h, e - (h - s)};
}

__device__ __forceinline__ F2 two_neg(F2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ F2 two_mul(F2 a, F2 b) {
    const float p = a.h * b.h;
    const float e = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
    const float h = p + e;
    return {h, e - (h - p)};
}
__device__ __forceinline__ F2 two_div(F2 a, F2 b) {
    const float q = a.h / b.h;
    const F2 r = two_add(a, two_neg(two_mul(F2{q, 0.f}, b)));
    const float q2 = r.h / b.h;
    const float h = q + q2;
    return {h, q2 - (h - q)};
}
// complex scalars of the recurrences: the FP64 pipe takes 64 cycles to issue a warp's instruction, and
// the hundred and fifty of an iteration (three divisions) cost more than its four hops
struct C2 {
    F2 re, im;
};
__device__ __forceinline__ C2 c2_mul(C2 a, C2 b) {
    return {two_add(two_mul(a.re, b.re), two_neg(two_mul(a.im, b.im))), two_add(two_mul(a.re, b.im), two_mul(a.im, b.re))};
}
__device__ __forceinline__ F2 c2_norm(C2 a) { return two_add(two_mul(a.re, a.re), two_mul(a.im, a.im)); }
__device__ __forceinline__ C2 c2_div(C2 a, C2 b, F2 bn) {   // bn = |b|^2
    const C2 n = c2_mul(a, C2{b.re, two_neg(b.im)});
    return {two_div(n.re, bn), two_div(n.im, bn)};
}
__device__ __forceinline__ float2 c2_round(C2 a) { return make_float2(a.re.h, a.im.h); }

struct SmallArgs {
    const int *nbr;          // [2][Vh][8]
    const float4 *L;         // [2][4][Vh][9] (re, re, im, im)
    const float *C;          // [2][Vh][2][72] clover inverse, (d, d) and (re, re, im, im)
    int Vh, nr;
    float hws, hwt;
    const c32 *b;            // [Vh][12][nr]
    c32 *x;                  // [Vh][12][nr]
    double rel_tol;
    int maxiter;
    int *iters, *status;     // [nr]
};

// psi of the neighbour times (1 -+ gamma_mu) U: half-spinor product k0, k1 and the signs of its lower part
template <bool FWD>
__device__ __forceinline__ void hop_half(int mu, const float2 *__restrict__ psi, const float4 *__restrict__ u, float c,
                                         float2 acc[12]) {
    float2 f[12];
    const float4 *q = reinterpret_cast<const float4 *>(psi);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float4 v = q[k];            // shared memory of a CTA of the cluster
        f[2 * k] = make_float2(v.x, v.y);
        f[2 * k + 1] = make_float2(v.z, v.w);
    }
    float2 h0[3], h1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {   // G d with G_1 = -i s1, G_2 = -i s2, G_3 = -i s3, G_4 = 1
        const float2 d0 = f[6 + a], d1 = f[9 + a];
        float2 g0 = mu == 0 ? cneg(ci(d1)) : mu == 1 ? cneg(d1) : mu == 2 ? cneg(ci(d0)) : d0;
        float2 g1 = mu == 0 ? cneg(ci(d0)) : mu == 1 ? d0 : mu == 2 ? ci(d1) : d1;
        h0[a] = FWD ? csub(f[a], g0) : cadd(f[a], g0);
        h1[a] = FWD ? csub(f[3 + a], g1) : cadd(f[3 + a], g1);
    }
    float2 k0[3], k1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) k0[a] = k1[a] = make_float2(0.f, 0.f);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float4 e = __ldg(u + a * 3 + b);
            const float2 m = make_float2(e.x, e.z);
            if (FWD) {
                k0[a] = cfma(m, h0[b], k0[a]);
                k1[a] = cfma(m, h1[b], k1[a]);
            } else {
                k0[b] = cfma_conj(m, h0[a], k0[b]);
                k1[b] = cfma_conj(m, h1[a], k1[b]);
            }
        }
    const float cl = FWD ? -c : c;
#pragma unroll
    for (int a = 0; a < 3; ++a) {   // lower = -+ G^dag k
        const float2 l0 = mu == 0 ? ci(k1[a]) : mu == 1 ? k1[a] : mu == 2 ? ci(k0[a]) : k0[a];
        const float2 l1 = mu == 0 ? ci(k0[a]) : mu == 1 ? cneg(k0[a]) : mu == 2 ? cneg(ci(k1[a])) : k1[a];
        acc[a] = make_float2(fmaf(c, k0[a].x, acc[a].x), fmaf(c, k0[a].y, acc[a].y));
        acc[3 + a] = make_float2(fmaf(c, k1[a].x, acc[3 + a].x), fmaf(c, k1[a].y, acc[3 + a].y));
        acc[6 + a] = make_float2(fmaf(cl, l0.x, acc[6 + a].x), fmaf(cl, l0.y, acc[6 + a].y));
        acc[9 + a] = make_float2(fmaf(cl, l1.x, acc[9 + a].x), fmaf(cl, l1.y, acc[9 + a].y));
    }
}

// A lane's two hops onto its site from the other parity: operands in the cluster's shared memory, links, weights
struct HopRef {
    const float2 *f, *b;
    const float4 *uf, *ub;
    float cf, cb;
};

// Components 3 mu .. 3 mu + 2 of A_pp^{-1} D in at site cb (all four lanes of the site call this)
__device__ __forceinline__ void hop_site(const SmallArgs &a, int p, int cb, int mu, const HopRef &r, float2 out[3]) {
    float2 acc[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = make_float2(0.f, 0.f);
    hop_half<true>(mu, r.f, r.uf, r.cf, acc);
    hop_half<false>(mu, r.b, r.ub, r.cb, acc);
    // lanes mu and mu ^ 2 keep one chirality each (spins 0, 1 in lanes 0, 1), then sum over mu ^ 1
    float2 x[6];
    const bool up = mu < 2;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float2 give = up ? acc[6 + k] : acc[k], keep = up ? acc[k] : acc[6 + k];
        x[k] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, give.x, 2), keep.y + __shfl_xor_sync(0xffffffffu, give.y, 2));
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        x[k].x += __shfl_xor_sync(0xffffffffu, x[k].x, 1);
        x[k].y += __shfl_xor_sync(0xffffffffu, x[k].y, 1);
    }
    // rows 3 (mu & 1) .. + 2 of the Hermitian block of this chirality
    const float *blk = a.C + (((long)p * a.Vh + cb) * 2 + (mu >> 1)) * 72;
    const float4 *lo = reinterpret_cast<const float4 *>(blk + 12);
    const int r0 = 3 * (mu & 1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int row = r0 + i;
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j == row) {
                const float d = __ldg(blk + 2 * row);
                s.x = fmaf(d, x[j].x, s.x);
                s.y = fmaf(d, x[j].y, s.y);
            } else {
                const float4 e = __ldg(lo + (row > j ? row * (row - 1) / 2 + j : j * (j - 1) / 2 + row));
                s = row > j ? cfma(make_float2(e.x, e.z), x[j], s) : cfma_conj(make_float2(e.x, e.z), x[j], s);
            }
        }
        out[i] = s;
    }
}

template <int T>
__global__ void __launch_bounds__(T) bicg_small_kernel(const SmallArgs a) {
    cg::cluster_group cluster = cg::this_cluster();
    const int nc = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int rhs = blockIdx.x / nc;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, mu = tid & 3;
    __shared__ F2 wsum[T / 32][SB_NRED];
    __shared__ F2 csum[2][SB_NRED];        // this CTA's sums, double-buffered over reductions
    __shared__ __align__(16) float2 us[T / 4][12], ws[T / 4][12];   // hop operands on this CTA's even and odd sites
    __shared__ F2 tot[SB_NRED];
    int cb = rank * (T / 4) + (tid >> 2);
    const bool in = cb < a.Vh;
    if (!in) cb = a.Vh - 1;                // works along with the warp, stores nothing
    HopRef ho[2];                          // onto the odd sites (from us) and onto the even ones (from ws)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int p = 1 - e;
        const int *nb = a.nbr + ((long)p * a.Vh + cb) * 8;
        const float wt = mu == 3 ? a.hwt : a.hws;
        const int jf = __ldg(nb + mu), jb = __ldg(nb + 4 + mu);
        const int nf = jf < 0 ? ~jf : jf, nk = jb < 0 ? ~jb : jb;
        float2(*buf)[12] = e == 0 ? us : ws;
        ho[e].f = cluster.map_shared_rank(&buf[nf % (T / 4)][0], nf / (T / 4));
        ho[e].b = cluster.map_shared_rank(&buf[nk % (T / 4)][0], nk / (T / 4));
        ho[e].uf = a.L + (((long)p * 4 + mu) * a.Vh + cb) * 9;
        ho[e].ub = a.L + (((long)(1 - p) * 4 + mu) * a.Vh + nk) * 9;
        ho[e].cf = jf < 0 ? -wt : wt;
        ho[e].cb = jb < 0 ? -wt : wt;
    }
    int red_no = 0;
    // sums of n reals over the cluster into tot[] (every CTA the same order); two barriers of the cluster
    // bracket it where the caller wants them: `publish` before one, `collect` after it
    auto publish = [&](F2 *v, int n) {
#pragma unroll
        for (int k = 0; k < SB_NRED; ++k) {
            if (k >= n) break;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const F2 t{__shfl_xor_sync(0xffffffffu, v[k].h, o), __shfl_xor_sync(0xffffffffu, v[k].l, o)};
                v[k] = two_add(v[k], t);
            }
            if (lane == 0) wsum[warp][k] = v[k];
        }
        __syncthreads();
        if (tid < n) {
            F2 s = wsum[0][tid];
            for (int q = 1; q < T / 32; ++q) s = two_add(s, wsum[q][tid]);
            csum[red_no & 1][tid] = s;
        }
    };
    auto collect = [&](int n) {
        if (warp == 0) {   // lane q reads CTA q's sums (at most 16 CTAs)
            F2 s[SB_NRED];
#pragma unroll
            for (int k = 0; k < SB_NRED; ++k) {
                s[k] = F2{0.f, 0.f};
                if (k < n && lane < nc) s[k] = *cluster.map_shared_rank(&csum[red_no & 1][k], lane);
            }
#pragma unroll
            for (int k = 0; k < SB_NRED; ++k) {
                if (k >= n) break;
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) {
                    const F2 t{__shfl_xor_sync(0xffffffffu, s[k].h, o), __shfl_xor_sync(0xffffffffu, s[k].l, o)};
                    s[k] = two_add(s[k], t);
                }
                if (lane == 0) tot[k] = s[k];
            }
        }
        ++red_no;
        __syncthreads();
    };

    float2 x[3], r[3], p[3], v[3], t[3];
    unsigned code = 0;
    F2 d[SB_NRED];
    auto zero_d = [&](int n) {
#pragma unroll
        for (int k = 0; k < SB_NRED; ++k)
            if (k < n) d[k] = F2{0.f, 0.f};
    };
    auto add_c = [&](int k, float2 z) {
        d[k] = two_add(d[k], F2{z.x, 0.f});
        d[k + 1] = two_add(d[k + 1], F2{z.y, 0.f});
    };
    auto rdot = [&](unsigned cd, float2 z) {   // conj(i^code) z
        const c32 y = rhat_conj_mul(cd & 3u, c32{z.x, z.y});
        return make_float2(y.re, y.im);
    };
    auto cdot = [&](float2 y, float2 z) { return make_float2(fmaf(y.y, z.y, y.x * z.x), fmaf(-y.y, z.x, y.x * z.y)); };
    auto put = [&](float2(*buf)[12], const float2 *f) {
        if (in) {
#pragma unroll
            for (int c = 0; c < 3; ++c) buf[tid >> 2][3 * mu + c] = f[c];
        }
    };

    // r = b, rhat = rounded phase of b, p = r; rho = <rhat, r>, rr = <r, r>
    zero_d(3);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const c32 z = a.b[((long)cb * 12 + 3 * mu + c) * a.nr + rhs];
        r[c] = in ? make_float2(z.re, z.im) : make_float2(0.f, 0.f);
        code |= rhat_quant(z.re, z.im) << (2 * c);
        p[c] = r[c];
        x[c] = make_float2(0.f, 0.f);
        add_c(0, rdot(code >> (2 * c), r[c]));
        d[2] = two_add(d[2], F2{fmaf(r[c].x, r[c].x, r[c].y * r[c].y), 0.f});
    }
    put(us, p);
    publish(d, 3);
    cluster.sync();
    collect(3);
    // every thread works the scalars out; state: 0 running, 1 converged, 2 breakdown, 3 no next direction
    C2 rho{tot[0], tot[1]};
    float rr = tot[2].h;
    const float stop = (float)(a.rel_tol * a.rel_tol) * rr;
    int its = 0;
    int state = (rr > 0.f && isfinite(rr) && c2_norm(rho).h > 0.f) ? 0 : rr > 0.f ? 2 : 1;
    F2 rsum{0.f, 0.f};   // this lane's part of <r, r>, summed with the next <rhat, v>

    while (state == 0 && its < a.maxiter) {
        ++its;
        // w = A_oo^{-1} D_oe p
        float2 h[3];
        hop_site(a, 1, cb, mu, ho[0], h);
        put(ws, h);
        cluster.sync();
        // v = p - A_ee^{-1} D_eo w, <rhat, v>, and <r, r> of the residual the iteration began with
        zero_d(3);
        d[2] = rsum;
        hop_site(a, 0, cb, mu, ho[1], h);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = in ? csub(p[c], h[c]) : make_float2(0.f, 0.f);
            add_c(0, rdot(code >> (2 * c), v[c]));
        }
        publish(d, 3);
        cluster.sync();
        collect(3);
        if (its > 1) rr = tot[2].h;
        const C2 dv{tot[0], tot[1]};
        const F2 dn = c2_norm(dv);
        if (!isfinite(rr))
            state = 2;
        else if (its > 1 && rr <= stop)
            state = 1;
        else if (!(dn.h > 0.f) || !isfinite(dn.h))
            state = 2;
        if (state != 0) {
            if (state == 1) --its;   // converged with the iteration before
            break;
        }
        const C2 alpha = c2_div(rho, dv, dn);
        // s = r - alpha v (in r)
        const float2 al = c2_round(alpha);
#pragma unroll
        for (int c = 0; c < 3; ++c) r[c] = cfma(cneg(al), v[c], r[c]);
        put(us, r);
        cluster.sync();
        // t = M s; <t, s>, <t, t>, <rhat, t>, <rhat, s>
        hop_site(a, 1, cb, mu, ho[0], h);
        put(ws, h);
        cluster.sync();
        zero_d(7);
        hop_site(a, 0, cb, mu, ho[1], h);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            t[c] = in ? csub(r[c], h[c]) : make_float2(0.f, 0.f);
            add_c(0, cdot(t[c], r[c]));
            add_c(2, rdot(code >> (2 * c), t[c]));
            add_c(4, rdot(code >> (2 * c), r[c]));
            d[6] = two_add(d[6], F2{fmaf(t[c].x, t[c].x, t[c].y * t[c].y), 0.f});
        }
        publish(d, 7);
        cluster.sync();
        collect(7);
        const F2 tt = tot[6], zero{0.f, 0.f};
        C2 omega{zero, zero}, beta{zero, zero};
        if (tt.h > 0.f && isfinite(tt.h))
            omega = C2{two_div(tot[0], tt), two_div(tot[1], tt)};   // else s = 0: the half step solved it
        const C2 ot = c2_mul(omega, C2{tot[2], tot[3]});
        const C2 rn{two_add(tot[4], two_neg(ot.re)), two_add(tot[5], two_neg(ot.im))};
        const C2 den = c2_mul(rho, omega);
        const F2 dq = c2_norm(den);
        if (dq.h > 0.f && isfinite(dq.h) && (rn.re.h != 0.f || rn.im.h != 0.f) && isfinite(rn.re.h) && isfinite(rn.im.h))
            beta = c2_div(c2_mul(rn, alpha), den, dq);   // (rn / rho)(alpha / omega)
        else
            state = 3;   // done if the residual is small, else a breakdown
        rho = rn;
        const float2 om = c2_round(omega), be = c2_round(beta);
        rsum = F2{0.f, 0.f};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[c] = cfma(om, r[c], cfma(al, p[c], x[c]));
            r[c] = cfma(cneg(om), t[c], r[c]);
            p[c] = cfma(be, cfma(cneg(om), v[c], p[c]), r[c]);
            rsum = two_add(rsum, F2{fmaf(r[c].x, r[c].x, r[c].y * r[c].y), 0.f});
        }
        put(us, p);
        if (state == 3 || its == a.maxiter) {   // the last residual's norm has no later reduction to go with
            zero_d(1);
            d[0] = rsum;
            publish(d, 1);
            cluster.sync();
            collect(1);
            state = tot[0].h <= stop ? 1 : state == 3 || !isfinite(tot[0].h) ? 2 : 0;
            break;
        }
        cluster.sync();
    }
    if (in) {
#pragma unroll
        for (int c = 0; c < 3; ++c) a.x[((long)cb * 12 + 3 * mu + c) * a.nr + rhs] = c32{x[c].x, x[c].y};
    }
    if (rank == 0 && tid == 0) {
        a.iters[rhs] = its;
        a.status[rhs] = state;
    }
    cluster.sync();   // no CTA leaves while another may still read its sums
}

template <int T>
void launch(const SmallArgs &a, int nc, cudaStream_t s) {
    LAPH_CUDA(cudaFuncSetAttribute(bicg_small_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.nr * nc));
    cfg.blockDim = dim3(T);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)nc;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LAPH_CUDA(cudaLaunchKernelEx(&cfg, bicg_small_kernel<T>, a));
    LAPH_LAUNCH_CHECK();
}

}  // namespace

// Shape of a right-hand side's cluster, and the blocks that are faster this way.  Measured with all
// else equal (whole solves, streamed / one kernel): 2^3 x 4 to 4^3 x 8 (T = 128) 2.1 to 3.3 up to 32
// right-hand sides and 1.7 to 2.4 at 64; 6^3 x 6 (16 CTAs of 256) 2.7, 2.0, 1.5 at 4, 8, 16 and 0.78 at
// 32; 8^3 x 8 (16 of 512) 2.2, 1.5, 1.15 at 4, 8, 16 and 0.64 at 32, 4^3 x 64 0.96 at 16: about seven
// clusters of 16 run at a time, the others wait for them.
static bool small_shape(long Vh, int nr, int &nc, int &T) {
    const long lanes = 4 * Vh;
    for (int t : {128, 256, 512})
        for (int c : {1, 2, 4, 8, 16}) {
            if ((long)t * c < lanes || (c < 8 && t > 128)) continue;
            nc = c;
            T = t;
            return nr <= (t == 512 ? 8 : t == 256 ? 16 : c == 16 ? 32 : 64);
        }
    return false;
}

bool bicg_small_fits(const DiracOp &op, int nr) {
    int nc, T;
    return small_shape(op.g.Vh, nr, nc, T);
}

void bicg_small(const DiracOp &op, int nr, const c32 *b, c32 *x, double rel_tol, int maxiter, int *iters,
                int *status, cudaStream_t s) {
    SmallArgs a;
    a.nbr = op.nbr;
    a.L = op.L32w;
    a.C = op.C32w;
    a.Vh = (int)op.g.Vh;
    a.nr = nr;
    a.hws = (float)op.hw[0];
    a.hwt = (float)op.hw[3];
    a.b = b;
    a.x = x;
    a.rel_tol = rel_tol;
    a.maxiter = maxiter;
    a.iters = iters;
    a.status = status;
    int nc = 1, T = 128;
    LAPH_REQUIRE(small_shape(op.g.Vh, nr, nc, T), "lattice too large for the one-kernel solver");
    if (T == 128)
        launch<128>(a, nc, s);
    else if (T == 256)
        launch<256>(a, nc, s);
    else
        launch<512>(a, nc, s);
}

}  // namespace laph
