// T_n(a (-Delta) + b) on the vectors of every slice in two-limb fixed point (fixed.cuh).
//
// The FP64 kernel (eigen.cu) needs 290 FP64 instructions per site at two lanes per cycle and SM: a warp
// takes 18000 cycles for it, so that even a 4^3 slice, one warp per scheduler, took 15 us a step.  Here a vector is kept through the whole chain as
// 58-bit integers over a power of two per site (cut once from FP64 at the start, rounded to FP64 once at
// the end): a step takes the largest exponent E of the site and its six neighbours, shifts their entries to
// it, and does the link products (648 IMAD.WIDE a site) and the recurrence with its coefficients in
// integers.  One thread per site: a thread per row would shift and split the 18 neighbour reals three times.
// A step of 4^3 x 16 or 6^3 x 8 takes 6.5 us (15.1), of 10^3 x 12 7.9 (15.7), of 16^3 x 32 34 with cold caches
// (95); N_v = 32 on 16^3 x 32, the whole call, 648 ms (859).
//
// Accuracy: entries are cut at 2^-58 of the largest in reach and sums rounded at 2^-57 of it, with the products of
// low limbs left out (rms 2^-57.3 a sum), against 2^-53 for every FP64 operation.  A site with NaN or infinities, and every site it reaches, becomes NaN.
#include <cmath>

#include "cheb_fix.cuh"
#include "fixed.cuh"

namespace laph {

namespace {

constexpr int EXP_NAN = 4096;   // a site with an entry that is not finite
constexpr double LINK_MAX = 1.0625;   // 36 products of a site stay below 2^62 in units 2^-56

__global__ void __launch_bounds__(128) links_kernel(long n, long V3, const c64 *__restrict__ U, int4 *__restrict__ out, int *flag) {
    const long i = (long)blockIdx.x * 128 + threadIdx.x;   // (t, x)
    if (i >= n) return;
    const long t = i / V3, x = i - t * V3;
    bool bad = false;
    for (int k = 0; k < 3; ++k)
        for (int e = 0; e < 9; ++e) {
            const c64 v = U[(i * 4 + k) * 9 + e];
            bad |= !(fabs(v.re) <= LINK_MAX && fabs(v.im) <= LINK_MAX);
            const FX r = to_fx(v.re), m = to_fx(v.im);
            out[((t * 3 + k) * 9 + e) * V3 + x] = make_int4(r.h, r.l, m.h, m.l);
        }
    if (bad) *flag = 1;
}

// vectors [t][v][x][3] to limb sums [q = t nvec + v][3][V3] and exponents [q][V3]
__global__ void __launch_bounds__(128) cut_vec_kernel(long V3, int nvec, long total, const c64 *__restrict__ in, long in_ts,
                                                      longlong2 *__restrict__ fix, short *__restrict__ exps) {
    const long i = (long)blockIdx.x * 128 + threadIdx.x;
    if (i >= total) return;
    const long q = i / V3, x = i - q * V3;
    const double2 *f = reinterpret_cast<const double2 *>(in) + (q / nvec) * in_ts + ((q % nvec) * V3 + x) * 3;
    double2 v[3];
    uint32_t m = 0, low = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        v[c] = __ldg(f + c);
        low |= (uint32_t)__double2loint(v[c].x) | (uint32_t)__double2loint(v[c].y);
        m = max(m, max((uint32_t)__double2hiint(v[c].x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(v[c].y) & 0x7FFFFFFFu));
    }
    const int ex = (int)(m >> 20);
    const int E = max(ex - 1022, EXP_MIN);
    exps[i] = (short)(ex == 0x7FF ? EXP_NAN : (m | low) == 0 ? EXP_NONE : E);
#pragma unroll
    for (int c = 0; c < 3; ++c) fix[(q * 3 + c) * V3 + x] = make_longlong2(cut(v[c].x, E), cut(v[c].y, E));
}

// D -= sum_j u_ij v_j (forward) or conj(u_ji) v_j (backward), v cut at 2^(E - sh - 58), D in units 2^(E - 56)
__device__ __forceinline__ void hop3(long long D[6], const longlong2 *__restrict__ f, const int4 *__restrict__ u, long V3, int sh,
                                     bool bwd) {
    CX v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const longlong2 z = __ldg(f + c * V3);
        v[c] = {limbs58(z.x >> sh), limbs58(z.y >> sh)};
    }
    const int si = bwd ? 1 : 3, sj = bwd ? 3 : 1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        Acc re, im;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int4 e = __ldg(u + (long)(i * si + j * sj) * V3);
            const FX ur{e.x, e.y}, ui = bwd ? FX{-e.z, -e.w} : FX{e.z, e.w};
            re.mad(ur, v[j].re);
            re.mad(neg(ui), v[j].im);
            im.mad(ur, v[j].im);
            im.mad(ui, v[j].re);
        }
        D[2 * i] -= floor_value(re);
        D[2 * i + 1] -= floor_value(im);
    }
}

// out = 2^twice (a (-Delta) + b) in - prev (PREV), as limb sums or, with LAST, in FP64
template <bool PREV, bool LAST>
__global__ void __launch_bounds__(64) cheb_fix_kernel(int ns, int V3, int nvec, long total, const int4 *__restrict__ links,
                                                      const longlong2 *__restrict__ in, const short *__restrict__ ein,
                                                      const longlong2 *__restrict__ prev, const short *__restrict__ eprev,
                                                      longlong2 *__restrict__ out, short *__restrict__ eout, c64 *__restrict__ dst,
                                                      long dst_ts, const int4 *__restrict__ ab, const int *__restrict__ abe,
                                                      int twice) {
    const long idx = (long)blockIdx.x * 64 + threadIdx.x;
    if (idx >= total) return;
    const long q = idx / V3;
    const int x = (int)(idx - q * V3), t = (int)(q / nvec), v = (int)(q - (long)t * nvec);
    const int cx = x % ns, r = x / ns, cy = r % ns, cz = r / ns;
    const short *ev = ein + q * V3;
    int nb[6], en[6];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int c = k == 0 ? cx : k == 1 ? cy : cz, st = k == 0 ? 1 : k == 1 ? ns : ns * ns;
        nb[2 * k] = c + 1 == ns ? x - st * (ns - 1) : x + st;
        nb[2 * k + 1] = c == 0 ? x + st * (ns - 1) : x - st;
    }
    const int es = ev[x];
    int E = max(es, EXP_MIN);
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        en[d] = ev[nb[d]];
        E = max(E, en[d]);
    }
    const int Ep = PREV ? eprev[q * V3 + x] : EXP_NONE;
    if (max(E, Ep) >= EXP_NAN) {
        const double nan = __longlong_as_double(0x7FF8000000000000ll);
        if constexpr (LAST)
            for (int c = 0; c < 3; ++c) dst[t * dst_ts + ((long)v * V3 + x) * 3 + c] = c64{nan, nan};
        else
            eout[q * V3 + x] = (short)EXP_NAN;
        return;
    }
    const longlong2 *f = in + q * 3 * V3;
    long long p[6], D[6];   // the site at E (units 2^-58), then 6 p - hops (units 2^-56)
    {
        const int sh = min(E - max(es, EXP_MIN - 64), 63);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const longlong2 z = __ldg(f + (long)c * V3 + x);
            p[2 * c] = z.x >> sh;
            p[2 * c + 1] = z.y >> sh;
        }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) D[c] = (6 * p[c] + 2) >> 2;
    const int4 *u = links + (long)t * 27 * V3;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        hop3(D, f + nb[2 * k], u + (long)k * 9 * V3 + x, V3, min(E - en[2 * k], 63), false);
        hop3(D, f + nb[2 * k + 1], u + (long)k * 9 * V3 + nb[2 * k + 1], V3, min(E - en[2 * k + 1], 63), true);
    }
    // a D + b p - prev at the exponent X: D with its leading bit at 2^57, at ed
    uint64_t any = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) any |= (uint64_t)(D[c] ^ (D[c] >> 63));
    const int up = min(__clzll((long long)any), 63) - 6;
    const int4 m = __ldg(ab + t);
    const int ec = __ldg(abe + t) + twice, e1 = E + 2 - up + ec, e2 = E + ec;
    const int X = max(max(e1, e2), Ep);
    const int s1 = min(X - e1, 62), s2 = min(X - e2, 62), s3 = min(X - Ep + 2, 62);
    const FX a{m.x, m.y}, b{m.z, m.w};
    long long y[6];
    any = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        Acc ta, tb;
        ta.mad(a, limbs58(up >= 0 ? D[c] << up : shr_near(D[c], -up)));
        tb.mad(b, limbs58(p[c]));
        y[c] = shr_near(ta.value(), s1) + shr_near(tb.value(), s2);
    }
    if constexpr (PREV) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const longlong2 z = __ldg(prev + (q * 3 + c) * V3 + x);
            y[2 * c] -= shr_near(z.x, s3);
            y[2 * c + 1] -= shr_near(z.y, s3);
        }
    }
    if constexpr (LAST) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            dst[t * dst_ts + ((long)v * V3 + x) * 3 + c] = c64{to_double(y[2 * c], X - 56), to_double(y[2 * c + 1], X - 56)};
    } else {
#pragma unroll
        for (int c = 0; c < 6; ++c) any |= (uint64_t)(y[c] ^ (y[c] >> 63));
        // |y| < 2^58: the leading bit to 2^57, units 2^-58 of 2^(X + 2 - uo)
        const int uo = max(min(__clzll((long long)any), 63) - 6, 0);
        bool zero = true;
#pragma unroll
        for (int c = 0; c < 6; ++c) zero &= y[c] == 0;
        eout[q * V3 + x] = (short)(zero ? EXP_NONE : X + 2 - uo);
#pragma unroll
        for (int c = 0; c < 3; ++c) out[(q * 3 + c) * V3 + x] = make_longlong2(y[2 * c] << uo, y[2 * c + 1] << uo);
    }
}

}  // namespace

void ChebMap::set(laph_ctx *ctx, const char *name, const std::vector<double> &a, const std::vector<double> &b, cudaStream_t s) {
    const size_t nt = a.size();
    ab = (int4 *)ws_get(ctx, (std::string(name) + ":ab").c_str(), sizeof(int4) * nt);
    e = (int *)ws_get(ctx, (std::string(name) + ":e").c_str(), sizeof(int) * nt);
    hab.assign(nt, make_int4(0, 0, 0, 0));
    he.assign(nt, 0);
    ok = true;
    auto limbs = [](double x, int ex, int &h, int &l) {   // x 2^-ex = h 2^-28 + l 2^-58
        const double y = std::ldexp(x, 28 - ex);
        h = (int)std::llrint(y);
        l = (int)std::llrint(std::ldexp(y - h, 30));
    };
    for (size_t t = 0; t < nt; ++t) {
        const double mx = std::max(std::fabs(a[t]), std::fabs(b[t]));
        if (!(std::isfinite(a[t]) && std::isfinite(b[t]) && mx > 1e-30 && mx < 1e30)) {
            ok = false;
            return;
        }
        he[t] = std::ilogb(mx) + 1;
        limbs(a[t], he[t], hab[t].x, hab[t].y);
        limbs(b[t], he[t], hab[t].z, hab[t].w);
    }
    LAPH_CUDA(cudaMemcpyAsync(ab, hab.data(), sizeof(int4) * nt, cudaMemcpyHostToDevice, s));
    LAPH_CUDA(cudaMemcpyAsync(e, he.data(), sizeof(int) * nt, cudaMemcpyHostToDevice, s));
}

void ChebFix::init(laph_ctx *c, const Geom &geom, const c64 *U, int nvec, cudaStream_t s) {
    ctx = c;
    g = geom;
    u = nullptr;
    if (g.V3 >= (1l << 30)) return;
    // vectors of a pass: three buffers of at most 256 MB (one vector of every slice at least)
    const size_t one = (size_t)g.V * 3 * sizeof(longlong2);
    chunk = (int)std::max(1l, std::min<long>(nvec, (256l << 20) / (long)one));
    longlong2 *buf = (longlong2 *)ws_spare(ctx, "cheb:f", 3 * one * chunk);
    int4 *w = (int4 *)ws_spare(ctx, "cheb:links", sizeof(int4) * 27 * g.V);
    if (!buf || !w) return;
    short *exps = (short *)ws_get(ctx, "cheb:e", 3 * sizeof(short) * g.V * (size_t)chunk);
    for (int i = 0; i < 3; ++i) {
        f[i] = buf + (size_t)i * 3 * g.V * chunk;
        e[i] = exps + (size_t)i * g.V * chunk;
    }
    int *flag = (int *)ws_get(ctx, "cheb:flag", sizeof(int));
    LAPH_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), s));
    links_kernel<<<grid_for(g.V, 128), 128, 0, s>>>(g.V, g.V3, U, w, flag);
    LAPH_LAUNCH_CHECK();
    int bad = 0;
    LAPH_CUDA(cudaMemcpyAsync(&bad, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
    LAPH_CUDA(cudaStreamSynchronize(s));
    if (!bad) u = w;
}

void ChebFix::chain(const ChebMap &m, int order, int nvec, const c64 *in, long in_ts, c64 *out, long out_ts,
                    cudaStream_t s) const {
    for (int v0 = 0; v0 < nvec; v0 += chunk) {
        const int nv = std::min(chunk, nvec - v0);
        const long total = (long)g.nt * nv * g.V3;
        cut_vec_kernel<<<grid_for(total, 128), 128, 0, s>>>(g.V3, nv, total, in + (long)v0 * 3 * g.V3, in_ts, f[0], e[0]);
        LAPH_LAUNCH_CHECK();
        c64 *dst = out + (long)v0 * 3 * g.V3;
        for (int k = 1; k <= order; ++k) {   // T_k in buffer k % 3
            const int i = (k + 2) % 3, p = (k + 1) % 3, o = k % 3;
            auto go = [&](auto kernel) {
                kernel<<<grid_for(total, 64), 64, 0, s>>>(g.ns, (int)g.V3, nv, total, u, f[i], e[i], f[p], e[p], f[o], e[o], dst,
                                                          out_ts, m.ab, m.e, k > 1 ? 1 : 0);
            };
            if (k == 1)
                k == order ? go(cheb_fix_kernel<false, true>) : go(cheb_fix_kernel<false, false>);
            else
                k == order ? go(cheb_fix_kernel<true, true>) : go(cheb_fix_kernel<true, false>);
            LAPH_LAUNCH_CHECK();
        }
    }
}

}  // namespace laph
