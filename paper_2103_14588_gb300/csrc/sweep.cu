// Crank-Nicolson sweep: a time-marching right preconditioner for flexible GMRES.
//
// The paper's conclusion (Sec. 5) asks for a preconditioner and points at
// decomposing the time direction.  Row t of D_w22 (Eq. 11) tests against the
// hat function of time node t, the sum of its halves on the elements (t-1, t)
// and (t, t+1).  Testing each time element against a constant instead gives
// Crank-Nicolson, the block lower-bidiagonal
//     B[t, t] = Bd = i M_s + (h_t/2) K_s,   B[t, t-1] = Bl = -i M_s + (h_t/2) K_s,
// with M_s the spatial mass matrix and K_s the spatial part of the operator
// (the sum of i alpha_k D^k - (m beta + V) D^0 over the spatial element
// matrices of Appendix A).  Averaging adjacent element rows, S = (I + U) / 2
// (U the shift to the next layer, the last layer keeping 1/2), reproduces the
// time derivative of D_w22 exactly and its spatial part up to a second
// difference in time.  The preconditioner is M = B^-1 S^-1:
//   s = S^-1 v:  s_{N-1} = 2 v_{N-1},  s_t = 2 v_t - s_{t+1}          (time scan)
//   x = B^-1 s:  x_0 = Bd^-1 s_0,      x_t = Bd^-1 (s_t - Bl x_{t-1}) (forward march)
// one spatial solve with Bd per layer.
//
// GPU layout of the work (FP32 vectors, the precision of the inner solve):
//   1. FFT over the periodic spatial axes of every (layer, x-node) plane, in
//      shared memory (mixed-radix Stockham);
//   2. s_0 = 2 sum_t (-1)^t v_t by one reading pass; the march then runs the time
//      scan forward, s_{t+1} = 2 v_t - s_t, beside the layer solves.  Per frequency:
//      spectral mode (every axis periodic, constant potential): M_s and K_s are
//        diagonal in frequency with 2 x 2 blocks, so the march is one scan over
//        t per frequency with a fixed recurrence;
//      banded mode (x Dirichlet, y / z periodic, potential depending on x only):
//        per frequency of (y, z) each layer solve is block tridiagonal along x,
//        solved by cyclic reduction with stored factors (sweep_march.cuh);
//   3. inverse FFT back to the node layout.
// The result is the same linear map as the assembled sweep (up to FP32
// rounding); meshes of other kinds (open axes, two or more non-periodic axes,
// a potential varying along a periodic axis) get DST_ERR_ARG.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "blas.h"
#include "internal.h"
#include "sweep.h"
#include "sweep_march.cuh"
#include "fft.cuh"

namespace {

constexpr double PI2 = 6.28318530717958647692;
constexpr int SWEEP_SMEM_LIMIT = 200 * 1024;     // dynamic shared memory of a CTA of the FFT and the march
using namespace dst_march;

// ---- 2a. spectral march: one thread per frequency ---------------------------
// Every axis periodic and a constant potential: M_s and K_s are diagonal in
// frequency with 2 x 2 blocks (1+1 and 2+1 only), so with P = Bd^-1 and M^ = prod_k m_k
//   x_t = P (s_t - Bl x_{t-1}) = x_{t-1} + P (s_t - h_t K^ x_{t-1})   (sweep_march.cuh),
// Bd = i M^ + (h_t/2) [ sum_k alpha_k (i sin th_k) i prod_{j != k} m_j - (m beta + V0) M^ ].
// The second form rounds relative to the increment.  LARGE: h_t K is not small against M
// (dst_sweep_plan's rule), s and h_t K x cancel, and the march takes
//   x_t = c x_{t-1} + P s_t - R x_{t-1},   R = Q + c I,   Q = P Bl = I - 2 i M^ P:
// -Q turns the two modes of a frequency by a phase each; c is the nearest of 1, -1, i, -i and 0 to
// that, exact, and R is formed in FP64, so the rounding is relative to R x.  Relative error of 48
// layers against FP64, at h_t = h, 10 h and 40 h (m = 1, V0 = 3, 24 x 24 nodes): 5.7e-7, 3.1e-7 and
// 2.8e-7 (the increment form 1.0e-6, 2.2e-6 and 4.1e-6); at h / 4 the increment form 4.7e-7, this
// one the same.  Either takes the same time.
// One pass over the layers, the loads of the next PD in flight while one is combined.
template <bool LARGE>
__global__ void march_spectral_kernel(SweepGeom g, const float4 *__restrict__ alt_hi,
                                      const float4 *__restrict__ alt_lo, float4 *__restrict__ x) {
    const int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t nf = (int64_t)g.n1 * g.n2;
    if (f >= nf) return;
    constexpr int PD = 8;
    float4 ring[PD];
#pragma unroll
    for (int q = 0; q < PD; ++q) ring[q] = q < g.nt ? x[q * nf + f] : make_float4(0.f, 0.f, 0.f, 0.f);
    // frequencies of the axes: FFT dims (outer n1, inner n2) map to physical axes ax1, ax2
    double th[3] = {0.0, 0.0, 0.0}, mk[2] = {1.0, 1.0};
    const int i1 = (int)(f / g.n2), i2 = (int)(f % g.n2);
    if (g.ax1 >= 0) th[g.ax1] = PI2 * i1 / g.n1;
    if (g.ax2 >= 0) th[g.ax2] = PI2 * i2 / g.n2;
    for (int k = 0; k < g.d; ++k) mk[k] = g.h[k] * (2.0 + cos(th[k])) / 3.0;
    const double pm = mk[0] * mk[1], ht2 = 0.5 * g.ht;
    const double bx = -ht2 * sin(th[0]) * mk[1], by = g.d > 1 ? -ht2 * sin(th[1]) * mk[0] : 0.0;
    // P, the inverse of [a0 + i pm, bx - i by; bx + i by, a1 + i pm]: (wx + i wy) = 1 / det
    const double a0 = -ht2 * (g.m + g.V0) * pm, a1 = -ht2 * (g.V0 - g.m) * pm;
    const double dx = a0 * a1 - pm * pm - (bx * bx + by * by), dy = pm * (a0 + a1), r = 1.0 / (dx * dx + dy * dy);
    const double wx = dx * r, wy = -dy * r;
    const double P[8] = {a1 * wx - pm * wy, a1 * wy + pm * wx, -bx * wx - by * wy, by * wx - bx * wy,
                         by * wy - bx * wx, -bx * wy - by * wx, a0 * wx - pm * wy, a0 * wy + pm * wx};
    auto blk = [](const double *v) {
        return Blk{make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]),
                   make_float4((float)v[4], (float)v[5], (float)v[6], (float)v[7])};
    };
    const Blk Pf = blk(P);
    // h_t K^ = kx sigma_x + ky sigma_y + diag(d0, d1)
    const float kx = (float)(2.0 * bx), ky = (float)(2.0 * by), d0 = (float)(-g.ht * (g.m + g.V0) * pm),
                d1 = (float)(-g.ht * (g.V0 - g.m) * pm);
    Blk Rf = {};
    float cx = 0.f, cy = 0.f;
    if (LARGE) {
        // Q by rows, then the c that leaves the smallest diagonal of R
        double Q[8];
#pragma unroll
        for (int k = 0; k < 8; k += 2) { Q[k] = 2.0 * pm * P[k + 1]; Q[k + 1] = -2.0 * pm * P[k]; }
        Q[0] += 1.0;
        Q[6] += 1.0;
        const float tx = (float)(Q[0] + Q[6]), ty = (float)(Q[1] + Q[7]);
        // |q0 + c|^2 + |q1 + c|^2 = |q0|^2 + |q1|^2 + 2 (|c|^2 + Re conj(c) (q0 + q1)): below that of c = 0 where the
        // trace has a part beyond -1 along c
        if (fmaxf(fabsf(tx), fabsf(ty)) > 1.f) {
            if (fabsf(tx) >= fabsf(ty)) cx = tx > 0.f ? -1.f : 1.f;
            else cy = ty > 0.f ? -1.f : 1.f;
        }
        Q[0] += cx; Q[6] += cx;
        Q[1] += cy; Q[7] += cy;
        Rf = blk(Q);
    }
    float4 s = alt_hi[f], lo = alt_lo[f], xp = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t t0 = 0; t0 < g.nt; t0 += PD) {
#pragma unroll
        for (int q = 0; q < PD; ++q) {
            const int64_t t = t0 + q;
            if (t < g.nt) {
                const float4 v = ring[q];
                if (t + PD < g.nt) ring[q] = x[(t + PD) * nf + f];
                float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
                if (LARGE) {
                    add_mv(u, Pf, add4(s, lo));
                    sub_mv(u, Rf, xp);
                    xp = make_float4(fmaf(cx, xp.x, fmaf(-cy, xp.y, u.x)), fmaf(cx, xp.y, fmaf(cy, xp.x, u.y)),
                                     fmaf(cx, xp.z, fmaf(-cy, xp.w, u.z)), fmaf(cx, xp.w, fmaf(cy, xp.z, u.w)));
                } else {
                    const float4 r =
                        make_float4(s.x - fmaf(kx, xp.z, fmaf(ky, xp.w, fmaf(d0, xp.x, -lo.x))),
                                    s.y - fmaf(kx, xp.w, fmaf(-ky, xp.z, fmaf(d0, xp.y, -lo.y))),
                                    s.z - fmaf(kx, xp.x, fmaf(-ky, xp.y, fmaf(d1, xp.z, -lo.z))),
                                    s.w - fmaf(kx, xp.y, fmaf(ky, xp.x, fmaf(d1, xp.w, -lo.w))));
                    add_mv(u, Pf, r);
                    xp = add4(u, xp);
                }
                x[t * nf + f] = xp;
                next_s(s, lo, v);
            }
        }
    }
}

}  // namespace

int dst_sweep_plan(const dst_mesh *mesh, SweepPlan &p) {
    std::memset(&p, 0, sizeof(p));
    const int d = mesh->d;
    int nonper = 0;
    for (int k = 0; k < d; ++k) {
        if (mesh->bc[k] == DST_BC_OPEN) {
            dst_internal_set_error_detail("Crank-Nicolson sweep: open axes are not supported");
            return DST_ERR_ARG;
        }
        if (mesh->bc[k] != DST_BC_PERIODIC) ++nonper;
    }
    if (nonper > 1 || (nonper == 1 && mesh->bc[0] != DST_BC_DIRICHLET)) {
        dst_internal_set_error_detail("Crank-Nicolson sweep: at most one non-periodic axis, and it must be x");
        return DST_ERR_ARG;
    }
    if (mesh->nt < 1) return DST_ERR_ARG;
    const bool banded = nonper == 1;
    // potential: constant on a spectral mesh, x-only on a banded one
    double V0 = 0.0;
    if (!mesh->V.empty()) {
        if (mesh->v_general) {
            dst_internal_set_error_detail("Crank-Nicolson sweep: the potential must depend on x only");
            return DST_ERR_ARG;
        }
        if (!banded) {
            V0 = mesh->V[0];
            for (int64_t e = 1; e < mesh->nel[0]; ++e)
                if (mesh->V[e] != V0) {
                    dst_internal_set_error_detail("Crank-Nicolson sweep: a potential varying along a periodic axis");
                    return DST_ERR_ARG;
                }
        }
    }
    SweepGeom &g = p.g;
    g.d = d;
    g.nc = mesh->nc;
    g.nt = mesh->nt;
    g.ht = mesh->ht;
    g.m = mesh->m;
    g.V0 = V0;
    for (int k = 0; k < 3; ++k) g.h[k] = mesh->h[k];
    g.nx = (int)mesh->nu[0];
    // FFT dims: the periodic axes, outer (n1) the slower one
    int per_axes[3], np = 0;
    for (int k = banded ? 1 : 0; k < d; ++k) per_axes[np++] = k;
    g.ax1 = g.ax2 = -1;
    g.n1 = g.n2 = 1;
    SweepFft &a = p.fft;
    a.nc = mesh->nc;
    a.nbx = banded ? (int)mesh->nu[0] : 1;
    a.sbx = 1;
    a.ns_nodes = mesh->n_spatial;
    int64_t stride[3] = {1, mesh->nu[0], mesh->nu[0] * mesh->nu[1]};
    if (np == 1) {
        g.ax2 = per_axes[0];
        g.n2 = (int)mesh->nu[per_axes[0]];
        a.s2 = stride[per_axes[0]];
        a.s1 = 0;
    } else if (np == 2) {
        g.ax2 = per_axes[0];
        g.ax1 = per_axes[1];
        g.n2 = (int)mesh->nu[per_axes[0]];
        g.n1 = (int)mesh->nu[per_axes[1]];
        a.s2 = stride[per_axes[0]];
        a.s1 = stride[per_axes[1]];
    } else if (np == 3) {
        dst_internal_set_error_detail("Crank-Nicolson sweep: a 3+1 mesh needs a Dirichlet x axis");
        return DST_ERR_ARG;
    }
    a.n1 = g.n1;
    a.n2 = g.n2;
    dst_fft::radices(a.n1, a.rad1, a.nrad1);
    dst_fft::radices(a.n2, a.rad2, a.nrad2);
    p.banded = banded;
    p.has_fft = np > 0;
    p.nb = banded ? mesh->nt * mesh->nu[0] : mesh->nt;
    const int64_t nf = (int64_t)g.n1 * g.n2;
    const int nmax = g.n1 > g.n2 ? g.n1 : g.n2;
    if (nmax > 4096) {
        dst_internal_set_error_detail("Crank-Nicolson sweep: a periodic axis longer than 4096 nodes");
        return DST_ERR_ARG;
    }
    const size_t limit = SWEEP_SMEM_LIMIT;
    if (p.has_fft && !dst_fft::choose_layout<float2>(a, p.nb, limit)) {
        dst_internal_set_error_detail("Crank-Nicolson sweep: a periodic plane too large for shared memory");
        return DST_ERR_ARG;
    }
    // h_t K against M: the derivatives, mass and potential (twice, as measured; both marches
    // give their errors on either side of the limits)
    double vmax = 0.0, kt = 2.0 * std::fabs(mesh->m);
    for (size_t e = 0; e < mesh->V.size() && e < (size_t)mesh->nel[0]; ++e) vmax = std::max(vmax, std::fabs(mesh->V[e]));
    kt += 2.0 * vmax;
    for (int k = 0; k < d; ++k) kt += 1.0 / mesh->h[k];
    p.large = g.ht * kt > (d == 1 ? 0.6 : 1.5) || g.ht > 0.5 * mesh->h[0];
    // banded march: G lanes per system (two x nodes each), `steps` parallel reduction
    // steps; systems per CTA as many as keep it at 256 threads while the CTAs still
    // cover the GPU (a 2+1 mesh has n_y systems, a 1+1 mesh one)
    if (banded) {
        if (g.nx > 365) {
            dst_internal_set_error_detail("Crank-Nicolson sweep: x axis too long for the banded march");
            return DST_ERR_ARG;
        }
        const int lanes = (g.nx + 1) / 2, npair = g.nc / 2;
        p.lanes = 8;
        while (p.lanes < lanes) p.lanes *= 2;
        p.steps = 0;
        while ((1 << p.steps) < lanes) ++p.steps;
        p.systems = 8;
        while (p.systems > npair && (p.systems * p.lanes > 256 || dst_march::march_smem(g.nc, p.systems, p.lanes, g.nx) > limit ||
                                     nf * npair < 152 * (int64_t)p.systems))
            p.systems /= 2;
        while (p.systems * p.lanes < 32) p.systems *= 2;       // whole warps
        p.march_smem = dst_march::march_smem(g.nc, p.systems, p.lanes, g.nx);
        if (p.march_smem > limit) {
            dst_internal_set_error_detail("Crank-Nicolson sweep: x axis too long for the banded march");
            return DST_ERR_ARG;
        }
        p.table_bytes = sizeof(float) * 8 * 2 * (size_t)dst_march::class_count(g.n1, g.n2) * dst_march::items(p.steps) * p.lanes;
    }
    p.launches = 2 + (p.has_fft ? 2 : 0);
    p.bytes_per_entry = 24.0 + (p.has_fft ? 32.0 : 0.0);
    p.vx = banded && !mesh->V.empty();
    return DST_OK;
}

static size_t pad256(size_t b) { return (b + 255) & ~(size_t)255; }

size_t dst_sweep_scratch_bytes(const SweepPlan &p, int64_t n_unknowns) {
    const size_t per = (size_t)(n_unknowns / p.g.nt);
    return pad256(sizeof(float2) * (size_t)n_unknowns) + pad256(p.table_bytes) +
           (p.banded ? pad256(sizeof(FreqRow) * (size_t)p.g.n1 * p.g.n2) : 0) + 2 * pad256(sizeof(float2) * per) +
           pad256((size_t)(p.g.nx + 2) * sizeof(double));
}

int dst_sweep_setup(const dst_mesh *mesh, SweepPlan &p, void *scratch, cudaStream_t s) {
    char *base = (char *)scratch;
    auto take = [&](size_t b) { char *at = base; base += pad256(b); return (void *)at; };
    const size_t per = (size_t)(mesh->n_unknowns / p.g.nt);
    const int nf = p.g.n1 * p.g.n2;
    p.work = (float2 *)take(sizeof(float2) * (size_t)mesh->n_unknowns);
    p.table = (float *)take(p.table_bytes);
    p.freq = p.banded ? (FreqRow *)take(sizeof(FreqRow) * (size_t)nf) : nullptr;
    p.alt_hi = (float4 *)take(sizeof(float2) * per);
    p.alt_lo = (float4 *)take(sizeof(float2) * per);
    p.dvx = p.vx ? (double *)take((size_t)(p.g.nx + 2) * sizeof(double)) : nullptr;
    if (p.vx)
        DST_CUDA_TRY(cudaMemcpyAsync(p.dvx, mesh->V.data(), sizeof(double) * mesh->nel[0], cudaMemcpyHostToDevice, s));
    if (p.banded) {
        const int per_cta = p.lanes < 64 ? 64 / p.lanes : 1, nsys = 2 * dst_march::class_count(p.g.n1, p.g.n2);
        const unsigned threads = (unsigned)(2 * per_cta * p.lanes);      // two per lane
        const unsigned blocks = (unsigned)((nsys + per_cta - 1) / per_cta + (nf + (int)threads - 1) / (int)threads);
        factor_kernel<<<blocks, threads, 3 * sizeof(M22) * (threads / 2), s>>>(p.g, p.lanes, p.steps, p.dvx, p.table, p.freq);
        DST_CUDA_TRY(cudaGetLastError());
    }
    return DST_OK;
}

template <int NC>
static int launch_march(const SweepPlan &p, const float2 *in, float2 *out, cudaStream_t s) {
    const int fper = NC == 4 ? p.systems / 2 : p.systems;
    const unsigned blocks = (unsigned)(((int64_t)p.g.n1 * p.g.n2 + fper - 1) / fper);
    auto go = [&](auto kern) -> int {
        // (the same limit for every plan: another thread may set it between this line and the launch)
        DST_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SWEEP_SMEM_LIMIT));
        kern<<<blocks, (unsigned)(p.systems * p.lanes), p.march_smem, s>>>(p.g, p.steps, p.dvx, p.table, p.freq, p.alt_hi,
                                                                          p.alt_lo, in, out);
        DST_CUDA_TRY(cudaGetLastError());
        return DST_OK;
    };
#define DST_MARCH(G) case G: return p.large ? go(march_kernel<NC, G, true>) : go(march_kernel<NC, G, false>);
    switch (p.lanes) {
        DST_MARCH(8) DST_MARCH(16) DST_MARCH(32) DST_MARCH(64) DST_MARCH(128) DST_MARCH(256)
        default: return DST_ERR_ARG;
    }
#undef DST_MARCH
}

// z = M v on FP32 vectors; p.work (n_unknowns float2) is the plan's scratch; v and z
// may not overlap it or each other.
int dst_sweep_apply(const SweepPlan &p, int64_t n_unknowns, const float2 *v, float2 *z, cudaStream_t s) {
    const int64_t per2 = n_unknowns / p.g.nt / 2;           // pairs of entries (NC is even)
    const int64_t nf = (int64_t)p.g.n1 * p.g.n2;
    // 1. forward FFT of every plane: v -> work (frequency layout); without an FFT the
    // march reads v and writes z
    const float2 *src = v;
    float2 *dst = z;
    // (the march wants 16-byte aligned layers: a vector that starts at an odd entry of its
    // buffer is marched in work too)
    const bool aside = !p.has_fft && (((uintptr_t)v | (uintptr_t)z) & 15) != 0;
    if (p.has_fft) {
        DST_CUDA_TRY((dst_fft::fft_launch<float2, false>(p.fft, p.nb, v, p.work, s)));
        src = dst = p.work;
    } else if (aside) {
        DST_CUDA_TRY(cudaMemcpyAsync(p.work, v, sizeof(float2) * n_unknowns, cudaMemcpyDeviceToDevice, s));
        src = dst = p.work;
    }
    // 2. s_0 and the march
    altsum_kernel<<<(unsigned)((per2 + 255) / 256), 256, 0, s>>>(per2, p.g.nt, (const float4 *)src, p.alt_hi, p.alt_lo);
    DST_CUDA_TRY(cudaGetLastError());
    if (!p.banded) {
        const auto march = p.large ? march_spectral_kernel<true> : march_spectral_kernel<false>;
        march<<<(unsigned)((nf + 63) / 64), 64, 0, s>>>(p.g, p.alt_hi, p.alt_lo, (float4 *)dst);
        DST_CUDA_TRY(cudaGetLastError());
    } else {
        const int rc = p.g.nc == 2 ? launch_march<2>(p, src, dst, s) : launch_march<4>(p, src, dst, s);
        if (rc) return rc;
    }
    // 3. inverse FFT: work -> z
    if (p.has_fft) DST_CUDA_TRY((dst_fft::fft_launch<float2, true>(p.fft, p.nb, p.work, z, s)));
    else if (aside) DST_CUDA_TRY(cudaMemcpyAsync(z, p.work, sizeof(float2) * n_unknowns, cudaMemcpyDeviceToDevice, s));
    return DST_OK;
}

extern "C" int dst_precond_apply(const dst_mesh *mesh, int kind, const void *v, void *z, void *stream) {
    if (!mesh || !v || !z || v == z) return DST_ERR_ARG;
    if (kind == DST_PRECOND_BLOCK_JACOBI) {
        cudaStream_t s = (cudaStream_t)stream;
        int rc = dst_internal_jacobi_setup(const_cast<dst_mesh *>(mesh), s);
        return rc ? rc : dst_internal_jacobi_apply(mesh, (const float2 *)v, (float2 *)z, s);
    }
    if (kind != DST_PRECOND_CN_SWEEP && kind != DST_PRECOND_CN_LEARNED) {
        dst_internal_set_error_detail("dst_precond_apply: unknown preconditioner kind");
        return DST_ERR_ARG;
    }
    if (kind == DST_PRECOND_CN_LEARNED && !dst_internal_unet_fits(mesh->unet, mesh)) {
        dst_internal_set_error_detail("dst_precond_apply: no network for this mesh (dst_set_learned_precond)");
        return DST_ERR_ARG;
    }
    SweepPlan p;
    int rc = dst_sweep_plan(mesh, p);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    void *scratch = nullptr;
    const int64_t n = mesh->n_unknowns;
    const size_t sweep_bytes = (dst_sweep_scratch_bytes(p, n) + 255) & ~(size_t)255;
    const size_t vec_bytes = ((size_t)n * sizeof(float2) + 255) & ~(size_t)255;
    const bool learned = kind == DST_PRECOND_CN_LEARNED;
    const bool aside = learned && ((uintptr_t)z & 15) != 0;       // the operator apply wants 16-byte aligned vectors
    const size_t bytes = sweep_bytes + (learned ? (aside ? 3 : 2) * vec_bytes : 0);
    if (cudaMallocAsync(&scratch, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return DST_ERR_OOM;
    }
    float2 *tmp = reinterpret_cast<float2 *>((char *)scratch + sweep_bytes);
    float2 *rho = reinterpret_cast<float2 *>((char *)tmp + vec_bytes);
    float2 *zz = aside ? reinterpret_cast<float2 *>((char *)rho + vec_bytes) : (float2 *)z;
    rc = dst_sweep_setup(mesh, p, scratch, s);
    if (rc == DST_OK) rc = dst_sweep_apply(p, n, (const float2 *)v, zz, s);
    if (rc == DST_OK && learned) {
        int nk = 0;
        rc = dst_internal_apply(mesh, DST_FP32, zz, tmp, s);                // rho = v - A M_CN(v)
        if (rc == DST_OK) rc = dst_k_sub_f32(n, (const float2 *)v, tmp, rho, s);
        if (rc == DST_OK) rc = dst_internal_unet_correct(mesh->unet, mesh, rho, zz, tmp, s, &nk);
        if (rc == DST_OK && aside && cudaMemcpyAsync(z, zz, sizeof(float2) * n, cudaMemcpyDeviceToDevice, s) != cudaSuccess)
            rc = DST_ERR_CUDA;
    }
    cudaFreeAsync(scratch, s);
    return rc;
}
