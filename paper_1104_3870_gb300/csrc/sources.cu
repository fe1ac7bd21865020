// Z4 noise in the LapH subspace and diluted sources (Sec. II, Eq. (varrhodef)
// with D = 1; dilution projectors P^(b) = P_T (x) P_S (x) P_L; Sec. IV noise).
//
// Noise: Philox4x32-10 (Salmon et al., SC'11) written from its definition:
// ten rounds of (hi0,lo0) = mulhilo(0xD2511F53, c0), (hi1,lo1) = mulhilo(0xCD9E8D57, c2),
// c <- (hi1^c1^k0, lo1, hi0^c3^k1, lo0), with the key bumped by
// (0x9E3779B9, 0xBB67AE85) before every round after the first.
// rho(t, alpha, n) = i^(w0 & 3) with counter ((t*4 + alpha)*nv + n, 0, 0, 0) and
// key ((config_id << 16) | noise_id, 0x4C415048).
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "philox.cuh"

namespace laph {

__global__ void z4_kernel(int n, uint32_t key0, uint8_t *codes) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t c[4] = {(uint32_t)i, 0u, 0u, 0u};
    philox4x32_10(c, key0, 0x4C415048u);
    codes[i] = (uint8_t)(c[0] & 3u);
}

void z4_codes(int nt, int nv, uint16_t noise_id, uint16_t config_id, uint8_t *codes, cudaStream_t s) {
    int n = nt * 4 * nv;
    uint32_t key0 = ((uint32_t)config_id << 16) | (uint32_t)noise_id;
    z4_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, key0, codes);
    LAPH_LAUNCH_CHECK();
}

// Projector diagonal of one dilution type (Sec. II table of schemes).
static bool proj(int type, int J, int N, int b, int i) {
    switch (type) {
        case 0: return true;
        case 1: return i == b;
        case 2: return (J * i) / N == b;
        default: return i % J == b;
    }
}

int n_proj(int type, int J, int N) {
    switch (type) {
        case 0: return 1;
        case 1: return N;
        case 2:
        case 3:
            LAPH_REQUIRE(J > 0 && N % J == 0, "dilution J must divide the dimension");
            return J;
        default: throw Error(LAPH_ERR_ARG, "unknown dilution type");
    }
}

// Host table mask[b][nt + 4 + nv] of the diagonals of P_T, P_S, P_L for each listed b.
std::vector<uint8_t> dilution_masks(const laph_dilution &d, int nt, int nv, const int *b_list, int nb) {
    int nT = n_proj(d.T.type, d.T.J, nt), nS = n_proj(d.S.type, d.S.J, 4), nL = n_proj(d.L.type, d.L.J, nv);
    int w = nt + 4 + nv;
    std::vector<uint8_t> m((size_t)nb * w);
    for (int i = 0; i < nb; ++i) {
        int b = b_list[i];
        LAPH_REQUIRE(b >= 0 && b < nT * nS * nL, "projector index out of range");
        int bL = b % nL, bS = (b / nL) % nS, bT = b / (nL * nS);
        for (int t = 0; t < nt; ++t) m[(size_t)i * w + t] = proj(d.T.type, d.T.J, nt, bT, t);
        for (int a = 0; a < 4; ++a) m[(size_t)i * w + nt + a] = proj(d.S.type, d.S.J, 4, bS, a);
        for (int n = 0; n < nv; ++n) m[(size_t)i * w + nt + 4 + n] = proj(d.L.type, d.L.J, nv, bL, n);
    }
    return m;
}

// out[b][site][alpha][c] = (gamma_4 y)_alpha,  y_alpha = sum_n V(t,n,x,c) [P^(b) rho](t,alpha,n).
// gamma_4 swaps the upper and lower spin pairs (chiral basis).
//
// Bound by the store of the result.  A block writes `sites` sites of one slice and projector: zeros in
// contiguous 16-byte stores where the time projector leaves the slice out (15 of 16 slices of (TI16, .)),
// else tile by tile through shared memory, from where they leave contiguously too.  (One thread per site and
// colour, storing four 16-byte pieces 48 bytes apart, reached 73 % of the copy bandwidth: half sectors.)  The
// vectors that the projector holds are listed once, so that a thread has eight of their entries in flight.
// 24^3 x 128, N_v = 64, 32 sources: 1.87 ms, 97 % of the copy bandwidth (1.92 ms without the list, 2.48 ms with one
// thread per site and colour); 12^3 x 16, 32 of 64 vectors in each of 16 sources: 185 us (338 and 201).
constexpr int SRC_SITES = 512, SRC_TILE = 64, SRC_THREADS = 192, SRC_LIST = 192;
__global__ void __launch_bounds__(SRC_THREADS) sources_kernel(long V3, int nt, int nv, int chunks, int sites,
                                                              const c64 *__restrict__ evecs,
                                                              const uint8_t *__restrict__ codes,
                                                              const uint8_t *__restrict__ mask, c64 *__restrict__ out) {
    const unsigned u = blockIdx.x / (unsigned)chunks, b = u / (unsigned)nt;   // (projector, slice)
    const int t = (int)(u - b * nt);
    const long x0 = (long)(blockIdx.x - u * chunks) * sites;
    const int ns = (int)min((long)sites, V3 - x0);
    const uint8_t *m = mask + (long)b * (nt + 4 + nv);
    double2 *o = reinterpret_cast<double2 *>(out) + ((long)u * V3 + x0) * 12;
    if (!m[t]) {
        const double2 z = make_double2(0.0, 0.0);
        for (int e = threadIdx.x; e < ns * 12; e += SRC_THREADS) o[e] = z;
        return;
    }
    __shared__ double2 sm[SRC_TILE * 12];
    __shared__ unsigned list[SRC_LIST];   // the projector's n among SRC_LIST, ascending: n << 8 | four 2-bit codes
    __shared__ int held[SRC_THREADS / 32];
    const int is = threadIdx.x / 3, c = threadIdx.x % 3, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool on[4] = {m[nt] != 0, m[nt + 1] != 0, m[nt + 2] != 0, m[nt + 3] != 0};
    auto build = [&](int n0) {
        const int n = n0 + (int)threadIdx.x;
        const bool in = n < nv && m[nt + 4 + n];
        unsigned w = (unsigned)n << 8;
        if (n < nv)
            for (int a = 0; a < 4; ++a) w |= (unsigned)codes[(t * 4 + a) * nv + n] << (2 * a);
        const unsigned who = __ballot_sync(0xffffffffu, in);
        if (lane == 0) held[warp] = __popc(who);
        __syncthreads();
        int first = 0, cnt = 0;
        for (int q = 0; q < SRC_THREADS / 32; ++q) {
            if (q < warp) first += held[q];
            cnt += held[q];
        }
        if (in) list[first + __popc(who & ((1u << lane) - 1))] = w;
        __syncthreads();
        return cnt;
    };
    int cnt = build(0);
    for (int s0 = 0; s0 < ns; s0 += SRC_TILE) {
        const int tile = min(SRC_TILE, ns - s0);
        c64 y[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
        for (int n0 = 0; n0 < nv; n0 += SRC_LIST) {
            if (nv > SRC_LIST && n0 + s0 > 0) {   // more vectors than a list holds
                __syncthreads();
                cnt = build(n0);
            }
            if (is >= tile) continue;
            const c64 *v = evecs + ((long)t * nv * V3 + x0 + s0 + is) * 3 + c;
            for (int i0 = 0; i0 < cnt; i0 += 8) {
                c64 vn[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (i0 + i < cnt) vn[i] = v[(long)(list[i0 + i] >> 8) * V3 * 3];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (i0 + i >= cnt) break;
                    const unsigned w = list[i0 + i];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        if (!on[a]) continue;
                        const unsigned code = (w >> (2 * a)) & 3u;
                        // i^code * vn
                        y[a] += code == 0 ? vn[i] : code == 1 ? times_i(vn[i]) : code == 2 ? -vn[i] : -times_i(vn[i]);
                    }
                }
            }
        }
        if (is < tile)
#pragma unroll
            for (int a = 0; a < 4; ++a) sm[is * 12 + a * 3 + c] = make_double2(y[(a + 2) & 3].re, y[(a + 2) & 3].im);
        __syncthreads();
        for (int e = threadIdx.x; e < tile * 12; e += SRC_THREADS) o[s0 * 12 + e] = sm[e];
        __syncthreads();
    }
}

// Sites of a block: 512 where that leaves every SM sixteen blocks with work, else down to one tile, since
// the tiles of a block follow one another (10^3 x 48, two sources: 39 us a call, 60 in blocks of 512 sites).
static int sources_sites(const laph_ctx *ctx, const Geom &g, const std::vector<uint8_t> &m, int nv, int nb) {
    long active = 0;   // (projector, slice) pairs that are not zero
    for (int b = 0; b < nb; ++b) {
        const uint8_t *q = m.data() + (size_t)b * (g.nt + 4 + nv);
        active += std::count(q, q + g.nt, (uint8_t)1);
    }
    int sites = SRC_SITES;
    while (sites > SRC_TILE && active * ((g.V3 + sites - 1) / sites) < 16l * (ctx->sm_count > 0 ? ctx->sm_count : 152)) sites /= 2;
    return sites;
}

}  // namespace laph

using namespace laph;

extern "C" int laph_make_sources(laph_ctx *ctx, const laph_lattice *lat, const void *evecs, int nv, uint16_t noise_id,
                                 uint16_t config_id, const laph_dilution *dil, const int *b_list, int nb, void *rhs,
                                 uint8_t *noise, void *stream) {
    return guard([&] {
        ctx_activate(ctx);
        Geom g = make_geom(lat);
        LAPH_REQUIRE(dil != nullptr, "dilution is null");
        LAPH_REQUIRE(nv >= 1 && nv <= 3 * g.V3, "nv out of range");
        LAPH_REQUIRE(nb >= 0, "nb must be >= 0");
        cudaStream_t s = as_stream(stream);
        std::vector<int> hb(nb);
        if (nb) {
            LAPH_REQUIRE(b_list != nullptr, "b_list is null");
            if (is_device_ptr(b_list)) {   // ordered on the caller's stream, then read on the host
                LAPH_CUDA(cudaMemcpyAsync(hb.data(), b_list, sizeof(int) * nb, cudaMemcpyDeviceToHost, s));
                LAPH_CUDA(cudaStreamSynchronize(s));
            } else
                std::copy(b_list, b_list + nb, hb.begin());
        }
        std::vector<uint8_t> m = dilution_masks(*dil, g.nt, nv, hb.data(), nb);
        size_t ebytes = sizeof(c64) * 3 * g.V3 * g.nt * (size_t)nv;
        const c64 *ev = (const c64 *)stage_in(ctx, evecs, ebytes, "evecs", s);
        uint8_t *codes = (uint8_t *)ws_get(ctx, "src:codes", (size_t)g.nt * 4 * nv);
        z4_codes(g.nt, nv, noise_id, config_id, codes, s);
        uint8_t *dm = (uint8_t *)ws_get(ctx, "src:mask", m.size() + 1);
        if (!m.empty()) LAPH_CUDA(cudaMemcpyAsync(dm, m.data(), m.size(), cudaMemcpyHostToDevice, s));
        size_t obytes = sizeof(c64) * 12 * g.V * (size_t)nb;
        StagedOut o = stage_out(ctx, rhs, obytes, "sources");
        if (nb) {
            const int sites = sources_sites(ctx, g, m, nv, nb);
            const int chunks = (int)((g.V3 + sites - 1) / sites);
            const int per = (int)std::max(1l, std::min<long>(nb, (1l << 30) / ((long)chunks * g.nt)));   // projectors a launch
            for (int b = 0; b < nb; b += per) {
                const int n = std::min(per, nb - b);
                sources_kernel<<<(unsigned)((long)chunks * g.nt * n), SRC_THREADS, 0, s>>>(
                    g.V3, g.nt, nv, chunks, sites, ev, codes, dm + (size_t)b * (g.nt + 4 + nv), (c64 *)o.dev + (size_t)b * g.V * 12);
                LAPH_LAUNCH_CHECK();
            }
        }
        if (noise) {
            StagedOut on = stage_out(ctx, noise, (size_t)g.nt * 4 * nv, "noise");
            LAPH_CUDA(cudaMemcpyAsync(on.dev, codes, (size_t)g.nt * 4 * nv, cudaMemcpyDeviceToDevice, s));
            on.commit(s);
        }
        o.commit(s);
        // keep the host mask alive until the async copy finished
        LAPH_CUDA(cudaStreamSynchronize(s));
    });
}
