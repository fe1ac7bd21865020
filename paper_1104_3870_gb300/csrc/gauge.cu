// Gauge preparation on the GPU: stout smearing (Sec. II).
#include <cmath>

#include "dirac.cuh"
#include "su3.cuh"

namespace laph {

// --------------------------------------------------------------------------
// Stout step.  One thread per (site, mu):
//   C = rho sum_{nu != mu} [U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag + U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)]
//   Omega = C U_mu^dag;  A = Omega^dag - Omega;  iQ = -A/2 + Tr(A)/6
//   U_mu <- exp(iQ) U_mu
// Reads `in`, writes `out` (all links of a step are updated simultaneously).
// --------------------------------------------------------------------------
__global__ void stout_kernel(Geom g, const c64 *__restrict__ in, c64 *__restrict__ out, double rho, int nmu) {
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.V * nmu) return;
    long s = idx / nmu;
    int mu = (int)(idx % nmu);
    int c[4];
    site_coords(g, s, c);
    int dims[4] = {g.ns, g.ns, g.ns, g.nt};
    auto shift = [&](const int *cc, int d, int step, int *o) {
        o[0] = cc[0]; o[1] = cc[1]; o[2] = cc[2]; o[3] = cc[3];
        o[d] = (cc[d] + step + dims[d]) % dims[d];
    };
    auto link = [&](const int *cc, int d) { return m3_load(in + (site_of(g, cc) * 4 + d) * 9); };
    M3 umu = link(c, mu);
    M3 csum = m3_zero();
    for (int nu = 0; nu < nmu; ++nu) {
        if (nu == mu) continue;
        int xp_nu[4], xp_mu[4], xm_nu[4], xm_nu_p_mu[4];
        shift(c, nu, 1, xp_nu);
        shift(c, mu, 1, xp_mu);
        shift(c, nu, -1, xm_nu);
        shift(xm_nu, mu, 1, xm_nu_p_mu);
        // upper staple
        M3 a = m3_mul(link(c, nu), link(xp_nu, mu));
        m3_add(csum, m3_mul_nd(a, link(xp_mu, nu)));
        // lower staple
        M3 unu_m = link(xm_nu, nu);
        M3 b = m3_mul_dn(unu_m, link(xm_nu, mu));
        m3_add(csum, m3_mul(b, link(xm_nu_p_mu, nu)));
    }
    M3 om = m3_scale(rho, m3_mul_nd(csum, umu));
    M3 x;
    double tr_im = 0.0;   // Tr(A) is purely imaginary for A anti-Hermitian
#pragma unroll
    for (int i = 0; i < 3; ++i) tr_im += -2.0 * om.m[i][i].im;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            c64 a = conj(om.m[j][i]) - om.m[i][j];   // A = Omega^dag - Omega
            x.m[i][j] = -0.5 * a;
        }
#pragma unroll
    for (int i = 0; i < 3; ++i) x.m[i][i].im += tr_im / 6.0;
    M3 e = m3_expm(x);
    m3_store(out + (s * 4 + mu) * 9, m3_mul(e, umu));
}

__global__ void copy_time_links(Geom g, const c64 *__restrict__ in, c64 *__restrict__ out) {
    long s = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.V) return;
#pragma unroll
    for (int k = 0; k < 9; ++k) out[(s * 4 + 3) * 9 + k] = in[(s * 4 + 3) * 9 + k];
}

}  // namespace laph

using namespace laph;

extern "C" int laph_stout_smear(laph_ctx *ctx, const laph_lattice *lat, void *links, double rho, int nsteps,
                                int spatial_only, void *stream) {
    return guard([&] {
        ctx_activate(ctx);
        Geom g = make_geom(lat);
        LAPH_REQUIRE(nsteps >= 0, "nsteps must be >= 0");
        cudaStream_t s = as_stream(stream);
        size_t bytes = sizeof(c64) * 9 * 4 * g.V;
        StagedOut out = stage_out(ctx, links, bytes, "stout_links");
        const void *in = stage_in(ctx, links, bytes, "stout_links_in", s);
        c64 *a = (c64 *)ws_get(ctx, "stout:a", bytes);
        c64 *b = (c64 *)ws_get(ctx, "stout:b", bytes);
        LAPH_CUDA(cudaMemcpyAsync(a, in, bytes, cudaMemcpyDeviceToDevice, s));
        int nmu = spatial_only ? 3 : 4;
        for (int k = 0; k < nsteps; ++k) {
            if (spatial_only) {
                copy_time_links<<<grid_for(g.V, 256), 256, 0, s>>>(g, a, b);
                LAPH_LAUNCH_CHECK();
            }
            stout_kernel<<<grid_for(g.V * nmu, 128), 128, 0, s>>>(g, a, b, rho, nmu);
            LAPH_LAUNCH_CHECK();
            std::swap(a, b);
        }
        LAPH_CUDA(cudaMemcpyAsync(out.dev, a, bytes, cudaMemcpyDeviceToDevice, s));
        out.commit(s);
    });
}
