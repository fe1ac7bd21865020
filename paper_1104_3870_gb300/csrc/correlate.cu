// Meson and I=2 two-pion correlators in LapH coefficient space (Sec. III,
// meson function Eq. (mesonfunc) at zero momentum without displacement, the
// connected term of Eq. (mesoncorr), gamma_5-swapped lines Eq. (laphpropg5)).
//
// For one quark line, the sink side is phi^[b](t,alpha,n) = coef (V_s^dag x) and
// the source side is rho^[b](t,alpha,n) = [P^(b) rho](t,alpha,n).  Because the
// eigenvectors of a slice are orthonormal, sum_{x,c} a(x)^* b(x) over LapH-smeared
// fields equals the same sum over LapH coordinates, so
//   M^[b1 b2](a, b; t) = sum_n sum_{alpha beta} conj(a^[b1](t,alpha,n)) W_{alpha beta} b^[b2](t,beta,n)
// with W = (gamma_5 gamma_4)^dag c for a barred first argument (rhobar adds a sign),
// c = gamma_4 Gamma.  The meson functions are FP64-accurate GEMMs on the tensor cores
// (mesonfn_tc.cu); the sums over projectors are FP64.
#include <cmath>
#include <vector>

#include "common.cuh"
#include "gamma_host.cuh"

namespace laph {

int n_proj(int type, int J, int N);   // sources.cu

// ----------------------------------------------------------------- kernels
// One projector diagonal of a dilution (Sec. II table of schemes).
__device__ __forceinline__ bool proj_at(int type, int J, int N, int b, int i) {
    return type == 0 ? true : type == 1 ? i == b : type == 2 ? (int)((long)J * i / N) == b : i % J == b;
}
__device__ __forceinline__ int proj_count(int type, int J, int N) { return type == 0 ? 1 : type == 1 ? N : J; }

// rho[line][b][alpha][n] = P^(b)(t0, alpha, n) i^code_line(t0, alpha, n) for up to four lines, with the
// projectors worked out here from the scheme (a host table of nb (nt + 4 + nv) bytes and its copy cost
// more than the kernel).
constexpr int RHO_BMAX = 512;
struct RhoLines {
    const uint8_t *codes[4];
    laph_dilution dil;
    const int *blist;   // device list, or null: b[]
    int b[RHO_BMAX];
};
__global__ void __launch_bounds__(256) rho_lines_kernel(const __grid_constant__ RhoLines a, int nt, int nv, int nb, int t0,
                                                        int nlines, c64 *__restrict__ out) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)nlines * nb * 4 * nv) return;
    const int n = (int)(idx % nv), al = (int)((idx / nv) % 4), i = (int)((idx / (4 * nv)) % nb);
    const int line = (int)(idx / ((long)4 * nv * nb));
    const int b = a.blist ? a.blist[i] : a.b[i];
    const int nS = proj_count(a.dil.S.type, a.dil.S.J, 4), nL = proj_count(a.dil.L.type, a.dil.L.J, nv);
    c64 v{0, 0};
    if (proj_at(a.dil.T.type, a.dil.T.J, nt, b / (nL * nS), t0) && proj_at(a.dil.S.type, a.dil.S.J, 4, (b / nL) % nS, al) &&
        proj_at(a.dil.L.type, a.dil.L.J, nv, b % nL, n)) {
        const int code = a.codes[line][(t0 * 4 + al) * nv + n];
        v = code == 0 ? c64{1, 0} : code == 1 ? c64{0, 1} : code == 2 ? c64{-1, 0} : c64{0, -1};
    }
    out[idx] = v;
}

// rho_src[b][alpha][n] = mask_b(t0,alpha,n) i^code(t0,alpha,n)
__global__ void rho_at_t0_kernel(int nt, int nv, int nb, int t0, const uint8_t *codes, const uint8_t *mask,
                                 c64 *out) {
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nb * 4 * nv) return;
    int b = idx / (4 * nv), a = (idx / nv) % 4, n = idx % nv;
    const uint8_t *m = mask + (long)b * (nt + 4 + nv);
    c64 v{0, 0};
    if (m[t0] && m[nt + a] && m[nt + 4 + n]) {
        int code = codes[(t0 * 4 + a) * nv + n];
        v = code == 0 ? c64{1, 0} : code == 1 ? c64{0, 1} : code == 2 ? c64{-1, 0} : c64{0, -1};
    }
    out[idx] = v;
}

// corr[dt] (+)= scale * sum_{b1 b2} M[t0+dt][b1][b2] conj(M[nt][b1][b2]): the connected correlator
// - sum M_sink conj(M_src) with M_src = -M[nt] (rhobar carries the sign).  M[z] has row stride ld; the
// block starts at element off.
__global__ void meson_contract_kernel(int nt, int nb, int ld, long off, int t0, const c64 *__restrict__ M, double scale,
                                      int add, c64 *corr) {
    __shared__ c64 sm[256];
    const int dt = blockIdx.x, t = (t0 + dt) % nt;
    const long zs = (long)ld * ld;
    const c64 *snk = M + t * zs + off, *src = M + nt * zs + off;
    c64 acc{0, 0};
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        const long i = (long)(e / nb) * ld + e % nb;
        acc += cmul_conj(src[i], snk[i]);
    }
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st) sm[threadIdx.x] += sm[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const c64 v = scale * sm[0];
        corr[dt] = add ? corr[dt] + v : v;
    }
}

__device__ __forceinline__ bool bits_zero(c64 s) {
    const long long b = __double_as_longlong(s.re) | __double_as_longlong(s.im);
    return (b << 1) == 0;
}
__device__ __forceinline__ bool bits_finite(c64 m) {
    return (__double2hiint(m.re) & 0x7FF00000) != 0x7FF00000 && (__double2hiint(m.im) & 0x7FF00000) != 0x7FF00000;
}

// X[t] = sum M14[b1][b4] M32[b3][b2] conj(S12[b1][b2]) conj(S34[b3][b4]) with both sources from M[nt] (their two
// signs cancel); M[z] holds rows (line 1, line 3) and columns (line 2, line 4).
// P[t][b1][b3] = sum_{b2} conj(S12[b1][b2]) M32[t][b3][b2]
__global__ void pipi_p_kernel(int nt, int nb, const c64 *__restrict__ M, c64 *__restrict__ P) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)nt * nb * nb) return;
    const int b3 = (int)(idx % nb), b1 = (int)((idx / nb) % nb), t = (int)(idx / ((long)nb * nb));
    const int ld = 2 * nb;
    const c64 *m = M + (long)t * ld * ld + (long)(nb + b3) * ld, *s12 = M + (long)nt * ld * ld + (long)b1 * ld;
    c64 s{0, 0};
    for (int b2 = 0; b2 < nb; ++b2) {
        const c64 a = s12[b2], v = m[b2];
        s += cmul_conj(a, v);
    }
    P[idx] = s;
}
// corr[dt] = cpi12 cpi34 - sum_{b1,b4} M14[t][b1][b4] sum_{b3} P[t][b1][b3] conj(S34[b3][b4])
__global__ void pipi_x_kernel(int nt, int nb, int t0, const c64 *__restrict__ P, const c64 *__restrict__ M,
                              const c64 *cpi12, const c64 *cpi34, c64 *corr) {
    __shared__ c64 sm[256];
    const int dt = blockIdx.x, t = (t0 + dt) % nt, ld = 2 * nb;
    const c64 *m14 = M + (long)t * ld * ld + nb, *s34 = M + (long)nt * ld * ld + (long)nb * ld + nb;
    const c64 *p = P + (long)t * nb * nb;
    c64 acc{0, 0};
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        const int b4 = e / nb, b1 = e % nb;
        c64 r{0, 0};
        for (int b3 = 0; b3 < nb; ++b3) {
            const c64 a = s34[(long)b3 * ld + b4], v = p[b1 * nb + b3];
            r += cmul_conj(a, v);
        }
        acc += m14[(long)b1 * ld + b4] * r;
    }
    sm[threadIdx.x] = acc;
    __syncthreads();
    for (int st = blockDim.x / 2; st > 0; st >>= 1) {
        if ((int)threadIdx.x < st) sm[threadIdx.x] += sm[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) corr[dt] = cpi12[dt] * cpi34[dt] - sm[0];
}

// The whole I = 2 pi pi correlator after the meson functions, one block per slice, for nb whose M32 and P
// matrices fit in shared memory: c12, c34 and X of pipi_x_kernel.  The sums run over lists of the nonzero
// source entries (one per row for full spin dilution): over all entries the FP64 pipe, two FMA per cycle
// and SM, bounds them at 57 + 62 us for nb = 32, nt = 128, even with the products predicated off.
__device__ __forceinline__ c64 block_sum256(c64 v, c64 *sm) {
    for (int o = 16; o > 0; o >>= 1) {
        v.re += __shfl_down_sync(0xffffffffu, v.re, o);
        v.im += __shfl_down_sync(0xffffffffu, v.im, o);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    c64 r{0, 0};
    for (int w = 0; w < (int)blockDim.x / 32; ++w) r += sm[w];
    return r;
}
__global__ void __launch_bounds__(512) pipi_slice_kernel(int nt, int nb, int t0, const c64 *__restrict__ M, c64 *corr) {
    extern __shared__ c64 psm[];
    __shared__ c64 red[16];
    const int dt = blockIdx.x, t = (t0 + dt) % nt, ld = 2 * nb, lp = nb + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long zs = (long)ld * ld;
    const c64 *m = M + t * zs, *src = M + nt * zs, *s34 = src + (long)nb * ld + nb;
    c64 *m32 = psm, *P = psm + nb * lp;
    // nonzero b2 of every row b1 of S12 and nonzero b3 of every column b4 of S34
    unsigned short *l12 = reinterpret_cast<unsigned short *>(P + nb * lp), *l34 = l12 + nb * nb, *n12 = l34 + nb * nb,
                   *n34 = n12 + nb;
    for (int r = warp; r < 2 * nb; r += blockDim.x / 32) {
        const bool first = r < nb;
        const int q = first ? r : r - nb;
        int n = 0;
        for (int k0 = 0; k0 < nb; k0 += 32) {
            const int k = k0 + lane;
            const bool nz = k < nb && !bits_zero(first ? src[(long)q * ld + k] : s34[(long)k * ld + q]);
            const unsigned mask = __ballot_sync(0xffffffffu, nz);
            if (nz) (first ? l12 : l34)[q * nb + n + __popc(mask & ((1u << lane) - 1))] = (unsigned short)k;
            n += __popc(mask);
        }
        if (lane == 0) (first ? n12 : n34)[q] = (unsigned short)n;
    }
    bool fin = true;
    c64 a12{0, 0}, a34{0, 0};
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        const int r = e / nb, k = e % nb;
        const c64 v = m[(long)(nb + r) * ld + k];
        m32[r * lp + k] = v;
        fin &= bits_finite(v);
        const long i = (long)r * ld + k, j = i + (long)nb * ld + nb;
        a12 += cmul_conj(src[i], m[i]);
        a34 += cmul_conj(src[j], m[j]);
    }
    const bool all2 = __syncthreads_or(!fin);   // a non-finite entry meets every element, zeros too
    fin = true;
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        const int b1 = e / nb, b3 = e % nb, n = all2 ? nb : n12[b1];
        const c64 *s12 = src + (long)b1 * ld, *v = m32 + b3 * lp;
        c64 s{0, 0};
        for (int i = 0; i < n; ++i) {
            const int b2 = all2 ? i : l12[b1 * nb + i];
            s += cmul_conj(s12[b2], v[b2]);
        }
        P[b1 * lp + b3] = s;
        fin &= bits_finite(s);
    }
    const bool all3 = __syncthreads_or(!fin);
    c64 x{0, 0};
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        const int b4 = e / nb, b1 = e % nb, n = all3 ? nb : n34[b4];
        const c64 *v = P + b1 * lp;
        c64 r{0, 0};
        for (int i = 0; i < n; ++i) {
            const int b3 = all3 ? i : l34[b4 * nb + i];
            r += cmul_conj(s34[(long)b3 * ld + b4], v[b3]);
        }
        x += m[(long)b1 * ld + nb + b4] * r;
    }
    a12 = block_sum256(a12, red);
    a34 = block_sum256(a34, red);
    x = block_sum256(x, red);
    if (threadIdx.x == 0) corr[dt] = a12 * a34 - x;
}

}  // namespace laph

using namespace laph;

extern "C" int correlate(laph_ctx *ctx, const laph_lattice *lat, const laph_corr_spec *spec, const void *const *coef,
                         const uint8_t *const *noise, void *corr, void *stream) {
    return guard([&] {
        ctx_activate(ctx);
        LAPH_REQUIRE(lat != nullptr && spec != nullptr && coef != nullptr && noise != nullptr, "null argument");
        const int nt = lat->nt, nv = spec->nv, nb = spec->nb, t0 = spec->t0;
        LAPH_REQUIRE(nt >= 1 && nv >= 1 && nb >= 1, "bad sizes");
        LAPH_REQUIRE(t0 >= 0 && t0 < nt, "t0 out of range");
        LAPH_REQUIRE(spec->b_list != nullptr, "b_list is null");
        int nlines = spec->channel == LAPH_CH_PIPI_I2 ? 4 : 2;
        LAPH_REQUIRE(spec->channel >= 0 && spec->channel <= LAPH_CH_PIPI_I2, "unknown channel");
        cudaStream_t s = as_stream(stream);
        const laph_dilution &dil = spec->dil;
        const long nproj = (long)n_proj(dil.T.type, dil.T.J, nt) * n_proj(dil.S.type, dil.S.J, 4) *
                           n_proj(dil.L.type, dil.L.J, nv);
        RhoLines rl{};
        rl.dil = dil;
        for (int i = 0; i < nb; ++i) {
            LAPH_REQUIRE(spec->b_list[i] >= 0 && spec->b_list[i] < nproj, "projector index out of range");
            if (nb <= RHO_BMAX) rl.b[i] = spec->b_list[i];
        }
        if (nb > RHO_BMAX) {
            int *d = (int *)ws_get(ctx, "corr:blist", sizeof(int) * nb);
            LAPH_CUDA(cudaMemcpyAsync(d, spec->b_list, sizeof(int) * nb, cudaMemcpyHostToDevice, s));
            rl.blist = d;
        }
        const c64 *cf[4] = {nullptr, nullptr, nullptr, nullptr};
        c64 *rho[4] = {nullptr, nullptr, nullptr, nullptr};
        for (int k = 0; k < nlines; ++k) {
            LAPH_REQUIRE(coef[k] != nullptr && noise[k] != nullptr, "line arrays are null");
            std::string id = std::to_string(k);
            cf[k] = (const c64 *)stage_in(ctx, coef[k], sizeof(c64) * (size_t)nb * nt * 4 * nv, "corr:coef" + id, s);
            rl.codes[k] = (const uint8_t *)stage_in(ctx, noise[k], (size_t)nt * 4 * nv, "corr:noise" + id, s);
        }
        const long per_line = (long)nb * 4 * nv;
        rho[0] = (c64 *)ws_get(ctx, "corr:rho", sizeof(c64) * nlines * per_line);
        for (int k = 1; k < nlines; ++k) rho[k] = rho[0] + k * per_line;
        rho_lines_kernel<<<grid_for(nlines * per_line, 256), 256, 0, s>>>(rl, nt, nv, nb, t0, nlines, rho[0]);
        LAPH_LAUNCH_CHECK();
        StagedOut out = stage_out(ctx, corr, sizeof(c64) * nt, "corr");
        c64 *c = (c64 *)out.dev;
        // rows: the barred lines (1 and, for pi pi, 3); columns: lines 2 and 4.  phibar = g5 g4 phi, so
        // W = (g5 g4)^dag c; one GEMM per W gives every sink function and, as slice nt, the sources
        const int nl = nlines / 2, ld = nl * nb;
        const MesonLines ml{nl, {cf[0], cf[2]}, {cf[1], cf[3]}, {rho[0], rho[2]}, {rho[1], rho[3]}};
        c64 *M = (c64 *)ws_get(ctx, "corr:M", sizeof(c64) * (size_t)(nt + 1) * ld * ld);
        const Mat4 g5g4d = mat_dag(mat_mul(gamma5(), gamma_mat(3)));
        if (nl == 1) {
            Mat4 cs[3];
            const int nc = channel_c(spec->channel, cs);
            for (int k = 0; k < nc; ++k) {
                meson_fns_tc(ctx, nt, nv, nb, ml, mat_mul(g5g4d, cs[k]), k == 0, M, s);
                meson_contract_kernel<<<nt, 256, 0, s>>>(nt, nb, ld, 0, t0, M, 1.0 / nc, k > 0, c);
                LAPH_LAUNCH_CHECK();
            }
        } else {
            meson_fns_tc(ctx, nt, nv, nb, ml, mat_mul(g5g4d, mat_mul(gamma_mat(3), gamma5())), true, M, s);
            const size_t shm = sizeof(c64) * 2 * (size_t)nb * (nb + 1) + sizeof(short) * 2 * ((size_t)nb * nb + nb);
            if (shm <= 220 * 1024) {   // nb <= 78
                LAPH_CUDA(cudaFuncSetAttribute(pipi_slice_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
                pipi_slice_kernel<<<nt, 512, shm, s>>>(nt, nb, t0, M, c);
                LAPH_LAUNCH_CHECK();
            } else {
                c64 *c12 = (c64 *)ws_get(ctx, "corr:c12", sizeof(c64) * nt);
                c64 *c34 = (c64 *)ws_get(ctx, "corr:c34", sizeof(c64) * nt);
                c64 *P = (c64 *)ws_get(ctx, "corr:P", sizeof(c64) * (size_t)nt * nb * nb);
                meson_contract_kernel<<<nt, 256, 0, s>>>(nt, nb, ld, 0, t0, M, 1.0, 0, c12);
                LAPH_LAUNCH_CHECK();
                meson_contract_kernel<<<nt, 256, 0, s>>>(nt, nb, ld, (long)nb * ld + nb, t0, M, 1.0, 0, c34);
                LAPH_LAUNCH_CHECK();
                pipi_p_kernel<<<grid_for((long)nt * nb * nb, 256), 256, 0, s>>>(nt, nb, M, P);
                LAPH_LAUNCH_CHECK();
                pipi_x_kernel<<<nt, 256, 0, s>>>(nt, nb, t0, P, M, c12, c34, c);
                LAPH_LAUNCH_CHECK();
            }
        }
        out.commit(s);
        LAPH_CUDA(cudaStreamSynchronize(s));
        xg::check_host_flag(ctx);
    });
}
