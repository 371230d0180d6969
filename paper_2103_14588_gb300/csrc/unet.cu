// Learned right preconditioner: a convolutional U-Net trained on the GPU.
//
// The paper names no preconditioner; its conclusion (Sec. 5) asks for one.  The
// network corrects the Crank-Nicolson sweep M_CN (sweep.cu):
//     M(v) = M_CN(v) + s U(rho / s),   rho = v - A M_CN(v),  s = ||rho||,
// so U is trained to map the sweep's residual to the sweep's error.  Training
// pairs come from the method itself: e random, r = A e (FP32 operator apply),
// z = M_CN(r), input rho = r - A z, target e - z (the exact solution of
// A d = rho), both divided by ||rho||; loss ||U(rho^) - t^||^2 / ||t^||^2; Adam.
//
// Network (three levels, 16 / 32 / 64 channels, C = 2 NC field channels, channel
// 2c = Re psi_c and 2c + 1 = Im psi_c, which is the complex unknown vector read as
// [node][channel] floats):
//   e1a conv3 C->16 ReLU, e1b conv3 16->16 ReLU = s1; pool;
//   e2a conv3 16->32 ReLU, e2b conv3 32->32 ReLU = s2; pool;
//   e3a conv3 32->64 ReLU, e3b conv3 64->64 ReLU; upsample;
//   u2p conv1 64->32, + s2, u2c conv3 32->32 ReLU; upsample;
//   u1p conv1 32->16, + s1, u1c conv3 16->16 ReLU; out conv1 16->C.
// pool = mean over 2^D blocks (cells past an odd end count as zero), upsample =
// nearest.  Convolutions run on BF16 tensor cores with FP32 accumulation
// (unet_kernels.cuh); parameters are kept in FP32 (Adam) and rounded to BF16.
// Parameter order and layout of the flat vector: per layer in the order above
// its weight (co, ci, kernel offsets row-major over the grid axes) then its bias.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "blas.h"
#include "internal.h"
#include "sweep.h"
#include "unet_kernels.cuh"

using namespace dst_nn;

namespace {

constexpr int NLAYER = 11;
enum { E1A, E1B, E2A, E2B, E3A, E3B, U2P, U2C, U1P, U1C, OUT };

struct Layer {
    int ci, co, taps, level;
    int kpad;               // K padded to 16
    int64_t woff, boff;     // offsets of weight and bias in the flat parameter vector
};

// Weights of every layer in fragment order (unet_kernels.cuh): wf for the forward pass, B[k][n] =
// W[n][c][tap] with k = tap * ci + c, and wt for the input gradient, the mirrored
// transpose B[k][n] = W[o][n][taps - 1 - tap] with k = tap * co + o.  The pair at
// [chunk][ntile][lane][h] holds k = 16 chunk + 8 h + 2 (lane % 4) and the next, n = 8 ntile + lane / 4.
struct PackLayer {
    int ci, co, taps;
    int nf, nt;                     // n tiles of wf and wt
    int64_t woff, first, count_f, count_t;   // weight offset; first pair of the layer; pairs of wf, wt
    uint32_t *wf, *wt;
};
struct PackLayers { PackLayer l[NLAYER]; int64_t total; };
__global__ void pack_weights_kernel(PackLayers P, const float *__restrict__ p) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= P.total) return;
    int l = 0;
    while (l + 1 < NLAYER && i >= P.l[l + 1].first) ++l;
    const PackLayer &L = P.l[l];
    int64_t at = i - L.first;
    const bool back = at >= L.count_f;
    if (back) at -= L.count_f;
    const int h = (int)(at & 1), lane = (int)((at >> 1) & 31), nt = back ? L.nt : L.nf;
    const int tile = (int)((at >> 6) % nt), chunk = (int)((at >> 6) / nt);
    const int n = tile * 8 + (lane >> 2), in = back ? L.co : L.ci, outs = back ? L.ci : L.co;
    float v[2];
    for (int e = 0; e < 2; ++e) {
        const int k = chunk * 16 + 8 * h + 2 * (lane & 3) + e, tap = k / in, c = k % in;
        v[e] = 0.f;
        if (n < outs && tap < L.taps)
            v[e] = back ? p[L.woff + ((int64_t)c * L.ci + n) * L.taps + (L.taps - 1 - tap)]
                        : p[L.woff + ((int64_t)n * L.ci + c) * L.taps + tap];
    }
    (back ? L.wt : L.wf)[at] = pack_bf16(v[0], v[1]);
}

__global__ void adam_kernel(int64_t n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                            float *__restrict__ v, float lr, float b1, float b2, float c1, float c2, float eps) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi, vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Sums of squares of one or two float arrays (blockIdx.y), one FP64 partial per CTA.
constexpr int SUM_CTAS = 456;
__global__ void __launch_bounds__(256) sumsq_kernel(int64_t n, const float *__restrict__ a, const float *__restrict__ b,
                                                    double *__restrict__ part) {
    __shared__ double red[256];
    const float *v = blockIdx.y ? b : a;
    double s = 0.0;
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < n; i += 256LL * gridDim.x) s += (double)v[i] * v[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.y * SUM_CTAS + blockIdx.x] = red[0];
}

// The sum of a sumsq_kernel's partials, the same in every CTA (one warp, fixed order).
__device__ __forceinline__ double total_of(const double *part, int count) {
    __shared__ double total;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int i = threadIdx.x; i < count; i += 32) s += part[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) total = s;
    }
    __syncthreads();
    const double t = total;
    __syncthreads();
    return t;
}

// The input scale s = ||x|| (a float scalar), and x / s in BF16 (n is even).
__global__ void __launch_bounds__(256) scale_input_kernel(int64_t n, int parts, const double *__restrict__ part,
                                                          const float2 *__restrict__ x, float *__restrict__ scale,
                                                          uint32_t *__restrict__ out) {
    const float s = (float)sqrt(total_of(part, parts)), inv = 1.0f / s;
    if (blockIdx.x == 0 && threadIdx.x == 0) *scale = s;
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < n / 2; i += 256LL * gridDim.x) {
        const float2 v = x[i];
        out[i] = pack_bf16(v.x * inv, v.y * inv);
    }
}

// dy = 2 (y - t / s) / ||t / s||^2 in BF16 with the column sums of its CTAs, and the
// CTAs' shares of ||y - t / s||^2; lq: log2 of the channels / 4.  t, a caller's vector, may
// start at any float.
__global__ void __launch_bounds__(256) loss_kernel(int64_t n4, int lq, int parts, const double *__restrict__ tpart,
                                                   const float4 *__restrict__ y, const float *__restrict__ t,
                                                   const float *__restrict__ s, uint2 *__restrict__ dy,
                                                   double *__restrict__ lpart, float *__restrict__ colsum) {
    __shared__ double red[256];
    const float inv = 1.0f / *s;
    const double tn = total_of(tpart, parts) * (double)inv * inv, w = 2.0 / tn;
    double acc = 0.0;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < n4; i += 256LL * gridDim.x) {
        const float4 a = y[i];
        const float4 r = make_float4(a.x - t[4 * i] * inv, a.y - t[4 * i + 1] * inv, a.z - t[4 * i + 2] * inv,
                                     a.w - t[4 * i + 3] * inv);
        acc += ((double)r.x * r.x + (double)r.y * r.y) + ((double)r.z * r.z + (double)r.w * r.w);
        const float4 d = make_float4((float)(w * r.x), (float)(w * r.y), (float)(w * r.z), (float)(w * r.w));
        dy[i] = pack_bf16x4(d);
        sum.x += d.x; sum.y += d.y; sum.z += d.z; sum.w += d.w;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) lpart[blockIdx.x] = red[0] / tn;
    cta_colsum(sum, lq, colsum);
}
__global__ void loss_sum_kernel(int parts, const double *__restrict__ lpart, double *__restrict__ loss) {
    const double t = total_of(lpart, parts);
    if (threadIdx.x == 0) *loss = t;
}

// <y, t / s> and ||y||^2 accumulated into acc[0], acc[1] (one CTA, FP64)
__global__ void dot_kernel(int64_t n, const float *__restrict__ y, const float *__restrict__ t,
                           const float *__restrict__ s, double *__restrict__ acc) {
    __shared__ double r1[256], r2[256];
    const float inv = 1.0f / *s;
    double a = 0.0, b = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        a += (double)y[i] * (double)(t[i] * inv);
        b += (double)y[i] * (double)y[i];
    }
    r1[threadIdx.x] = a;
    r2[threadIdx.x] = b;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) { r1[threadIdx.x] += r1[threadIdx.x + w]; r2[threadIdx.x] += r2[threadIdx.x + w]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { acc[0] += r1[0]; acc[1] += r2[0]; }
}

// Partial sums of <a, r> = sum conj(a_i) r_i (re, im) and ||a||^2 over complex
// vectors, one triple per CTA (FP64), for the least-squares scale of the correction.
constexpr int LS_PARTS = 304;
__global__ void __launch_bounds__(256) ls_partials_kernel(int64_t n, const float2 *__restrict__ a,
                                                          const float2 *__restrict__ r, double *__restrict__ part) {
    __shared__ double red[3][256];
    double re = 0.0, im = 0.0, aa = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 ai = a[i], ri = r[i];
        re += (double)ai.x * ri.x + (double)ai.y * ri.y;
        im += (double)ai.x * ri.y - (double)ai.y * ri.x;
        aa += (double)ai.x * ai.x + (double)ai.y * ai.y;
    }
    red[0][threadIdx.x] = re; red[1][threadIdx.x] = im; red[2][threadIdx.x] = aa;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < 3; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 3) part[3 * blockIdx.x + threadIdx.x] = red[threadIdx.x][0];
}

// z += alpha y with alpha = <a, r> / ||a||^2 from the partials (0 when a = 0);
// every CTA sums the partials in the same order, so all use the same alpha.
__global__ void __launch_bounds__(256) ls_axpy_kernel(int64_t n, int nparts, const double *__restrict__ part,
                                                      const float2 *__restrict__ y, float2 *__restrict__ z) {
    __shared__ float2 alpha;
    if (threadIdx.x == 0) {
        double re = 0.0, im = 0.0, aa = 0.0;
        for (int b = 0; b < nparts; ++b) { re += part[3 * b]; im += part[3 * b + 1]; aa += part[3 * b + 2]; }
        alpha = aa > 0.0 ? make_float2((float)(re / aa), (float)(im / aa)) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        const float2 yi = y[i];
        float2 zi = z[i];
        zi.x += alpha.x * yi.x - alpha.y * yi.y;
        zi.y += alpha.x * yi.y + alpha.y * yi.x;
        z[i] = zi;
    }
}

// standard normal pairs from splitmix64 of (seed, index) by Box-Muller
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__global__ void randn_kernel(int64_t n, uint64_t seed, float2 *__restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t a = mix64(seed ^ mix64((uint64_t)i));
    const double u1 = ((a >> 11) + 1.0) * (1.0 / 9007199254740993.0);
    const double u2 = (mix64(a) >> 11) * (1.0 / 9007199254740992.0);
    const double r = sqrt(-2.0 * log(u1));
    double sn, cs;
    sincospi(2.0 * u2, &sn, &cs);
    out[i] = make_float2((float)(r * cs), (float)(r * sn));
}

inline unsigned nblk(int64_t n) { return (unsigned)((n + 255) / 256); }

}  // namespace

struct dst_unet {
    int device;
    int d, nc, C;
    UGrid grid[3];
    Layer L[NLAYER];
    int64_t nparams;
    float *params, *grads, *adam_m, *adam_v;     // FP32 [nparams]
    PackLayers pack;                             // weight fragments
    GradLayers sums;                             // partial sums of the weight and bias gradients
    float *wpart, *bpart;
    bf16 *zeros;                                 // 64 channels of zeros: a node outside the grid
    // activations [N][ch]: BF16 where only a convolution (or a ReLU mask) reads them
    bf16 *x0, *a1, *p1, *a2, *p2, *a3, *h3, *q2, *r2, *q1, *r1;
    float *s1, *s2, *y;
    bf16 *z1, *z2;                               // gradients that a convolution reads (the widest layer each)
    float *gs1, *gs2, *gup;                      // gradients of s1, s2, and before an adjoint
    float *scale;                                          // device scalar s
    float *gamma;                                          // device scalar: output scale of the correction
    double gamma_host;
    double *dscr;                                          // device doubles: [1] loss, [2], [3] sums over fresh pairs
    double *spart;                                         // partial sums of squares and of the loss (3 x SUM_CTAS)
    double *part;                                          // LS_PARTS x 3 partial sums of the correction's scale
    void *mem;
    size_t mem_bytes;
    bool packed;
};

static UGrid coarse(const UGrid &f) {
    UGrid c;
    c.D = f.D;
    c.N = 1;
    for (int a = 0; a < f.D; ++a) {
        c.n[a] = (f.n[a] + 1) / 2;
        c.N *= c.n[a];
    }
    for (int a = f.D; a < 4; ++a) c.n[a] = 1;
    return c;
}

// ---- launch shapes ----------------------------------------------------------

// Weight gradients, kernel 3: segments of an x line (up to 64 nodes), and slices so that
// the CTAs (three or nine warps each) fill the GPU twice while the slices stay within
// two million partial sums; kernel 1: 32 nodes at a time, one slice per warp.  Loss and gradients at
// 48^3: 586, 565 and 565 us with 152, 304 and 608 CTAs for 16 channels, 621, 564 and 560 us with
// 2^20, 2^21 and 2^22 partial sums (8 MB a layer at 2^21); at 64^3 846, 815, 811 and 913, 812, 793.
static int wgrad_seg(const UGrid &g) {
    const int nx = g.n[g.D - 1], segs = (nx + WG_MAX_SEG - 1) / WG_MAX_SEG;
    return (nx + segs - 1) / segs;
}
static int wgrad_items(const Layer &L, const UGrid &g) {
    if (L.taps == 1) return (int)((g.N + 31) / 32);
    const int nx = g.n[g.D - 1];
    return (int)(g.N / nx * ((nx + wgrad_seg(g) - 1) / wgrad_seg(g)));
}
static int wgrad_slices(const Layer &L, const UGrid &g) {
    const int items = wgrad_items(L, g);
    const int64_t dw = (int64_t)L.co * L.kpad, most = std::max<int64_t>(1, (2 << 20) / dw);
    if (L.taps == 1) return (int)std::min<int64_t>((items + 3) / 4 * 4, 4 * std::min<int64_t>(152, std::max<int64_t>(1, most / 4)));
    return (int)std::min<int64_t>(items, std::min<int64_t>(std::max(1, 304 * 16 / L.co), most));
}
// Rows of column sums a layer's bias gradient may take (one per CTA that produces its dz).
static int64_t colsum_rows(const UGrid &g) { return std::max<int64_t>((g.N + 16 * CONV_WARPS - 1) / (16 * CONV_WARPS), SUM_CTAS); }
// CTAs of an element-wise kernel with column sums
static unsigned sum_ctas(int64_t quads) { return (unsigned)std::min<int64_t>(SUM_CTAS, (quads + 255) / 256); }

static int unet_create(const dst_mesh *mesh, dst_unet **out) {
    dst_unet *u = new (std::nothrow) dst_unet();
    if (!u) return DST_ERR_OOM;
    std::memset(u, 0, sizeof(*u));
    DST_CUDA_TRY(cudaGetDevice(&u->device));
    u->d = mesh->d;
    u->nc = mesh->nc;
    u->C = 2 * mesh->nc;
    UGrid &g1 = u->grid[0];
    g1.D = mesh->d + 1;
    g1.n[0] = (int)mesh->nt;
    for (int a = 1; a < g1.D; ++a) g1.n[a] = (int)mesh->nu[mesh->d - a];     // t, [z], [y], x
    for (int a = g1.D; a < 4; ++a) g1.n[a] = 1;
    g1.N = mesh->nt * mesh->n_spatial;
    u->grid[1] = coarse(g1);
    u->grid[2] = coarse(u->grid[1]);
    int taps3 = 1;
    for (int a = 0; a < g1.D; ++a) taps3 *= 3;
    const int spec[NLAYER][4] = {{-1, 16, 3, 0}, {16, 16, 3, 0}, {16, 32, 3, 1}, {32, 32, 3, 1}, {32, 64, 3, 2},
                                 {64, 64, 3, 2}, {64, 32, 1, 1}, {32, 32, 3, 1}, {32, 16, 1, 0}, {16, 16, 3, 0},
                                 {16, -1, 1, 0}};
    int64_t off = 0;
    for (int l = 0; l < NLAYER; ++l) {
        Layer &L = u->L[l];
        L.ci = spec[l][0] < 0 ? u->C : spec[l][0];
        L.co = spec[l][1] < 0 ? u->C : spec[l][1];
        L.taps = spec[l][2] == 3 ? taps3 : 1;
        L.level = spec[l][3];
        L.kpad = (L.taps * L.ci + 15) / 16 * 16;
        L.woff = off;
        off += (int64_t)L.co * L.ci * L.taps;
        L.boff = off;
        off += L.co;
    }
    u->nparams = off;
    // one device allocation for everything
    const int64_t N1 = g1.N, N2 = u->grid[1].N, N3 = u->grid[2].N;
    size_t total = 0;
    auto take = [&](size_t b) { size_t o = total; total += (b + 255) & ~(size_t)255; return o; };
    const size_t o_par = take(4 * sizeof(float) * u->nparams);
    size_t o_wf[NLAYER], o_wt[NLAYER];
    int64_t pairs = 0, wfloats = 0, bfloats = 0, cells = 0;
    for (int l = 0; l < NLAYER; ++l) {
        const Layer &L = u->L[l];
        PackLayer &P = u->pack.l[l];
        P.ci = L.ci; P.co = L.co; P.taps = L.taps; P.woff = L.woff;
        P.nf = (L.co + 7) / 8; P.nt = (L.ci + 7) / 8;
        P.count_f = (int64_t)(L.kpad / 16) * P.nf * 64;
        P.count_t = l == E1A ? 0 : (int64_t)((L.taps * L.co + 15) / 16) * P.nt * 64;
        P.first = pairs;
        pairs += P.count_f + P.count_t;
        o_wf[l] = take(sizeof(uint32_t) * P.count_f);
        o_wt[l] = take(sizeof(uint32_t) * P.count_t);
        GradLayer &G = u->sums.l[l];
        G.co = L.co; G.ci = L.ci; G.taps = L.taps; G.kpad = L.kpad; G.woff = L.woff; G.boff = L.boff;
        G.slices = wgrad_slices(L, u->grid[L.level]);
        G.wpart = wfloats; G.bpart = bfloats; G.first = cells;
        wfloats += (int64_t)G.slices * L.co * L.kpad;
        bfloats += colsum_rows(u->grid[L.level]) * L.co;
        cells += (int64_t)L.co * L.kpad;
    }
    u->pack.total = pairs;
    u->sums.n = NLAYER;
    u->sums.total = cells;
    const size_t o_zero = take(sizeof(bf16) * 64);
    const size_t o_wp = take(sizeof(float) * wfloats), o_bp = take(sizeof(float) * bfloats);
    const int64_t half[] = {N1 * u->C, N1 * 16, N2 * 16, N2 * 32, N3 * 32, N3 * 64, N3 * 64, N2 * 32, N2 * 32, N1 * 16, N1 * 16};
    size_t o_half[11];
    for (int k = 0; k < 11; ++k) o_half[k] = take(sizeof(bf16) * half[k]);
    const int64_t wide = std::max(std::max(N1 * 16, N2 * 32), N3 * 64), up = std::max(N1 * 32, N2 * 64);
    const size_t o_z1 = take(sizeof(bf16) * wide), o_z2 = take(sizeof(bf16) * wide);
    const size_t o_s1 = take(sizeof(float) * N1 * 16), o_s2 = take(sizeof(float) * N2 * 32);
    const size_t o_y = take(sizeof(float) * N1 * u->C);
    const size_t o_gs1 = take(sizeof(float) * N1 * 16), o_gs2 = take(sizeof(float) * N2 * 32), o_gup = take(sizeof(float) * up);
    const size_t o_sc = take(sizeof(float) * 4), o_ds = take(sizeof(double) * 4);
    const size_t o_sp = take(sizeof(double) * 3 * SUM_CTAS);
    const size_t o_pt = take(sizeof(double) * 3 * LS_PARTS);
    if (cudaMalloc(&u->mem, total) != cudaSuccess) {
        cudaGetLastError();
        delete u;
        return DST_ERR_OOM;
    }
    u->mem_bytes = total;
    char *b = (char *)u->mem;
    u->params = (float *)(b + o_par);
    u->grads = u->params + u->nparams;
    u->adam_m = u->grads + u->nparams;
    u->adam_v = u->adam_m + u->nparams;
    for (int l = 0; l < NLAYER; ++l) {
        u->pack.l[l].wf = (uint32_t *)(b + o_wf[l]);
        u->pack.l[l].wt = (uint32_t *)(b + o_wt[l]);
    }
    u->zeros = (bf16 *)(b + o_zero);              // (the allocation is cleared below)
    u->wpart = (float *)(b + o_wp);
    u->bpart = (float *)(b + o_bp);
    bf16 **half_p[11] = {&u->x0, &u->a1, &u->p1, &u->a2, &u->p2, &u->a3, &u->h3, &u->q2, &u->r2, &u->q1, &u->r1};
    for (int k = 0; k < 11; ++k) *half_p[k] = (bf16 *)(b + o_half[k]);
    u->z1 = (bf16 *)(b + o_z1);
    u->z2 = (bf16 *)(b + o_z2);
    u->s1 = (float *)(b + o_s1);
    u->s2 = (float *)(b + o_s2);
    u->y = (float *)(b + o_y);
    u->gs1 = (float *)(b + o_gs1);
    u->gs2 = (float *)(b + o_gs2);
    u->gup = (float *)(b + o_gup);
    u->scale = (float *)(b + o_sc);
    u->gamma = u->scale + 1;
    u->dscr = (double *)(b + o_ds);
    u->spart = (double *)(b + o_sp);
    u->part = (double *)(b + o_pt);
    cudaError_t e = cudaMemset(u->mem, 0, total);
    const float one = 1.0f;
    if (e == cudaSuccess) e = cudaMemcpy(u->gamma, &one, sizeof(float), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(u->mem);
        delete u;
        DST_CUDA_TRY(e);
    }
    u->gamma_host = 1.0;
    *out = u;
    return DST_OK;
}

static int pack(dst_unet *u, cudaStream_t s) {
    pack_weights_kernel<<<nblk(u->pack.total), 256, 0, s>>>(u->pack, u->params);
    DST_CUDA_TRY(cudaGetLastError());
    u->packed = true;
    return DST_OK;
}

// Channels of output per warp (8 NT) and rows (16 MT): the widest tile that leaves eight
// warps per SM, because a wide tile loads its operands less often (forward at 48^3: 156, 154, 155
// and 160 us with 4, 8, 16 and 32).
static int launch_conv(const ConvArgs &a, unsigned *ctas, cudaStream_t s) {
    const int64_t want = 152 * 8, tiles = (a.g.N + 15) / 16;
    int nt = std::min(a.ntiles, 4), mt = 2;
    while (mt * nt > 1 && (tiles + mt - 1) / mt * (a.ntiles / nt) < want) {
        if (mt > 1) mt = 1;
        else nt /= 2;
    }
    const dim3 grid((unsigned)((tiles + CONV_WARPS * mt - 1) / (CONV_WARPS * mt)), (unsigned)(a.ntiles / nt));
    if (ctas) *ctas = grid.x;
    int rc = DST_OK;
    auto launch = [&](auto n_, auto m_, auto c_) {
        constexpr int NT = decltype(n_)::value, MT = decltype(m_)::value, C = decltype(c_)::value;
        const size_t smem = C > 0 ? ConvShape<NT, MT, C == 0 ? 1 : C>::SMEM : 0;
        auto kern = conv_kernel<NT, MT, C>;
        if (smem > 40 * 1024 &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            rc = DST_ERR_CUDA;
        else
            kern<<<grid, 32 * CONV_WARPS, smem, s>>>(a);
    };
    auto go = [&](auto c16) {
        using I1 = std::integral_constant<int, 1>;
        using I2 = std::integral_constant<int, 2>;
        using I4 = std::integral_constant<int, 4>;
        if (nt == 4) { if (mt == 2) launch(I4(), I2(), c16); else launch(I4(), I1(), c16); }
        else if (nt == 2) { if (mt == 2) launch(I2(), I2(), c16); else launch(I2(), I1(), c16); }
        else { if (mt == 2) launch(I1(), I2(), c16); else launch(I1(), I1(), c16); }
    };
    // a kernel of one tap has nothing to stage ahead (32 -> 16 channels at 48^3: 10 us, 19 staged)
    switch (a.taps == 1 ? 2 : a.lci) {
        case 2: case 3: go(std::integral_constant<int, 0>()); break;
        case 4: go(std::integral_constant<int, 1>()); break;
        case 5: go(std::integral_constant<int, 2>()); break;
        case 6: go(std::integral_constant<int, 4>()); break;
        default: return DST_ERR_ARG;
    }
    DST_CUDA_TRY(cudaGetLastError());
    return rc;
}

static int log2i(int v) {
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

struct ConvOut {
    float *f32 = nullptr;                   // FP32 and / or BF16 result
    bf16 *b16 = nullptr;
    const float *res = nullptr;             // added before the activation
    bool relu = false;
    const bf16 *mask = nullptr;             // ReLU mask of a gradient
    const float *s1 = nullptr, *s2 = nullptr;
};

// layer l on `in`, read at each node's parent in the next coarser grid if `from_coarse`
static int conv(dst_unet *u, int l, const bf16 *in, const ConvOut &o, cudaStream_t s, bool from_coarse = false) {
    const Layer &L = u->L[l];
    ConvArgs a = {};
    a.g = u->grid[L.level];
    a.coarse = from_coarse ? 1 : 0;
    if (from_coarse) a.up = u->grid[L.level + 1];
    a.lci = log2i(L.ci); a.taps = L.taps; a.chunks = L.kpad / 16; a.co = L.co; a.ntiles = u->pack.l[l].nf;
    a.in = in; a.zeros = u->zeros; a.w = u->pack.l[l].wf; a.bias = u->params + L.boff; a.res = o.res; a.relu = o.relu ? 1 : 0;
    a.s1 = o.s1; a.s2 = o.s2; a.out32 = o.f32; a.out16 = o.b16;
    return launch_conv(a, nullptr, s);
}

// input gradient of layer l: dx[n][ci] = sum dz[n - off][co] W[co][ci][tap]; `next`: the
// layer whose dz the masked result is (its bias gradient takes the column sums), or -1
static int conv_dgrad(dst_unet *u, int l, const bf16 *dz, const ConvOut &o, int next, cudaStream_t s) {
    const Layer &L = u->L[l];
    ConvArgs a = {};
    a.g = u->grid[L.level];
    a.lci = log2i(L.co); a.taps = L.taps; a.chunks = (L.taps * L.co + 15) / 16; a.co = L.ci; a.ntiles = u->pack.l[l].nt;
    a.in = dz; a.zeros = u->zeros; a.w = u->pack.l[l].wt;                   // mirrored taps
    a.mask = o.mask; a.out32 = o.f32; a.out16 = o.b16;
    unsigned rows = 0;
    if (next >= 0) a.colsum = u->bpart + u->sums.l[next].bpart;
    const int rc = launch_conv(a, &rows, s);
    if (next >= 0) u->sums.l[next].rows = (int)rows;
    return rc;
}

static int conv_wgrad(dst_unet *u, int l, const bf16 *in, const bf16 *dz, cudaStream_t s, bool from_coarse = false) {
    const Layer &L = u->L[l];
    const UGrid &g = u->grid[L.level];
    WgradArgs a = {};
    a.g = g; a.ci = L.ci; a.taps = L.taps; a.kpad = L.kpad; a.co = L.co;
    a.coarse = from_coarse ? 1 : 0;
    if (from_coarse) a.up = u->grid[L.level + 1];
    a.in = in; a.dz = dz; a.dw = u->wpart + u->sums.l[l].wpart;
    a.seg = wgrad_seg(g);
    a.segs = (g.n[g.D - 1] + a.seg - 1) / a.seg;
    a.items = wgrad_items(L, g);
    const int slices = u->sums.l[l].slices;
    a.per_cta = (a.items + slices - 1) / slices;
    const unsigned rows16 = (unsigned)((L.co + 15) / 16);
    if (L.taps == 1) {
        const dim3 grid((unsigned)(slices / 4), rows16);
        switch (L.ci) {
            case 16: wgrad1_kernel<2><<<grid, 128, 0, s>>>(a); break;
            case 32: wgrad1_kernel<4><<<grid, 128, 0, s>>>(a); break;
            case 64: wgrad1_kernel<8><<<grid, 128, 0, s>>>(a); break;
            default: return DST_ERR_ARG;
        }
    } else {
        const int offsets = L.taps / 3, warps = std::min(offsets, 9);
        const dim3 grid((unsigned)slices, rows16, (unsigned)(offsets / warps));
        auto go = [&](auto kern, int ci8) -> int {
            const size_t smem = 2 * wg_buffer(ci8, warps, a.seg);
            // (the kernel's largest: another thread's mesh may set it between this line and the launch)
            DST_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)(2 * wg_buffer(ci8, 9, WG_MAX_SEG))));
            kern<<<grid, 32 * warps, smem, s>>>(a);
            return DST_OK;
        };
        int rc;
        switch (L.ci) {
            case 4: case 8: rc = go(wgrad3_kernel<1>, 1); break;
            case 16: rc = go(wgrad3_kernel<2>, 2); break;
            case 32: rc = go(wgrad3_kernel<4>, 4); break;
            case 64: rc = go(wgrad3_kernel<8>, 8); break;
            default: return DST_ERR_ARG;
        }
        if (rc) return rc;
    }
    DST_CUDA_TRY(cudaGetLastError());
    return DST_OK;
}

// s = ||x|| into u->scale and x / s into u->x0; with a target also the partial sums of its square
static int set_input(dst_unet *u, const float *x, const float *target, cudaStream_t s) {
    const int64_t n = u->grid[0].N * u->C;
    const unsigned parts = sum_ctas(n / 4);
    sumsq_kernel<<<dim3(parts, target ? 2 : 1), 256, 0, s>>>(n, x, target, u->spart);
    scale_input_kernel<<<(unsigned)std::min<int64_t>(608, (n / 2 + 255) / 256), 256, 0, s>>>(
        n, (int)parts, u->spart, (const float2 *)x, u->scale, (uint32_t *)u->x0);
    DST_CUDA_TRY(cudaGetLastError());
    return DST_OK;
}

// U(x0) on the node grid, stored as `out` says
static int forward(dst_unet *u, const ConvOut &out, cudaStream_t s) {
    int rc;
    if (!u->packed && (rc = pack(u, s))) return rc;
    const UGrid &g1 = u->grid[0], &g2 = u->grid[1], &g3 = u->grid[2];
    auto relu16 = [](bf16 *b) { ConvOut o; o.b16 = b; o.relu = true; return o; };
    auto relu32 = [](float *f) { ConvOut o; o.f32 = f; o.relu = true; return o; };
    auto plus = [](bf16 *b, const float *res) { ConvOut o; o.b16 = b; o.res = res; return o; };
    if ((rc = conv(u, E1A, u->x0, relu16(u->a1), s))) return rc;
    if ((rc = conv(u, E1B, u->a1, relu32(u->s1), s))) return rc;
    pool_kernel<<<nblk(g2.N * 4), 256, 0, s>>>(g1, g2, 2, (const float4 *)u->s1, (uint2 *)u->p1);
    if ((rc = conv(u, E2A, u->p1, relu16(u->a2), s))) return rc;
    if ((rc = conv(u, E2B, u->a2, relu32(u->s2), s))) return rc;
    pool_kernel<<<nblk(g3.N * 8), 256, 0, s>>>(g2, g3, 3, (const float4 *)u->s2, (uint2 *)u->p2);
    if ((rc = conv(u, E3A, u->p2, relu16(u->a3), s))) return rc;
    if ((rc = conv(u, E3B, u->a3, relu16(u->h3), s))) return rc;
    if ((rc = conv(u, U2P, u->h3, plus(u->q2, u->s2), s, true))) return rc;
    if ((rc = conv(u, U2C, u->q2, relu16(u->r2), s))) return rc;
    if ((rc = conv(u, U1P, u->r2, plus(u->q1, u->s1), s, true))) return rc;
    if ((rc = conv(u, U1C, u->q1, relu16(u->r1), s))) return rc;
    return conv(u, OUT, u->r1, out, s);
}
constexpr int FORWARD_LAUNCHES = 13;

// gradients of every parameter (into u->grads, overwritten); dL/dy is in u->z1 and its
// column sums in the partials of OUT
static int backward(dst_unet *u, cudaStream_t s) {
    const UGrid &g1 = u->grid[0], &g2 = u->grid[1], &g3 = u->grid[2];
    bf16 *z = u->z1, *zn = u->z2;
    int rc;
    // dz of layer l from the gradient at its input's producer: masked by y, BF16
    auto masked = [](bf16 *b, const bf16 *y) { ConvOut o; o.b16 = b; o.mask = y; return o; };
    auto both = [](bf16 *b, float *f) { ConvOut o; o.b16 = b; o.f32 = f; return o; };
    auto plain = [](float *f) { ConvOut o; o.f32 = f; return o; };
    auto next = [&] { std::swap(z, zn); };
    auto colsum = [&](int l, unsigned ctas) {
        u->sums.l[l].rows = (int)ctas;
        return u->bpart + u->sums.l[l].bpart;
    };
    if ((rc = conv_wgrad(u, OUT, u->r1, z, s))) return rc;
    if ((rc = conv_dgrad(u, OUT, z, masked(zn, u->r1), U1C, s))) return rc;
    next();
    if ((rc = conv_wgrad(u, U1C, u->q1, z, s))) return rc;
    if ((rc = conv_dgrad(u, U1C, z, both(zn, u->gs1), U1P, s))) return rc;         // d q1 = d s1
    next();
    if ((rc = conv_wgrad(u, U1P, u->r2, z, s, true))) return rc;
    if ((rc = conv_dgrad(u, U1P, z, plain(u->gup), -1, s))) return rc;             // d (upsampled r2)
    unsigned ctas = sum_ctas(g2.N * 8);
    up_adjoint_kernel<<<ctas, 256, 0, s>>>(g1, g2, 3, (const float4 *)u->gup, (const uint2 *)u->r2, (uint2 *)zn, colsum(U2C, ctas));
    next();
    if ((rc = conv_wgrad(u, U2C, u->q2, z, s))) return rc;
    if ((rc = conv_dgrad(u, U2C, z, both(zn, u->gs2), U2P, s))) return rc;         // d q2 = d s2
    next();
    if ((rc = conv_wgrad(u, U2P, u->h3, z, s, true))) return rc;
    if ((rc = conv_dgrad(u, U2P, z, plain(u->gup), -1, s))) return rc;             // d (upsampled h3)
    ctas = sum_ctas(g3.N * 16);
    up_adjoint_kernel<<<ctas, 256, 0, s>>>(g2, g3, 4, (const float4 *)u->gup, (const uint2 *)u->h3, (uint2 *)zn, colsum(E3B, ctas));
    next();
    if ((rc = conv_wgrad(u, E3B, u->a3, z, s))) return rc;
    if ((rc = conv_dgrad(u, E3B, z, masked(zn, u->a3), E3A, s))) return rc;
    next();
    if ((rc = conv_wgrad(u, E3A, u->p2, z, s))) return rc;
    if ((rc = conv_dgrad(u, E3A, z, plain(u->gup), -1, s))) return rc;             // d p2
    ctas = sum_ctas(g2.N * 8);
    pool_adjoint_kernel<<<ctas, 256, 0, s>>>(g2, g3, 3, (const float4 *)u->gs2, (const float4 *)u->gup, (const float4 *)u->s2,
                                             (uint2 *)zn, colsum(E2B, ctas));
    next();
    if ((rc = conv_wgrad(u, E2B, u->a2, z, s))) return rc;
    if ((rc = conv_dgrad(u, E2B, z, masked(zn, u->a2), E2A, s))) return rc;
    next();
    if ((rc = conv_wgrad(u, E2A, u->p1, z, s))) return rc;
    if ((rc = conv_dgrad(u, E2A, z, plain(u->gup), -1, s))) return rc;             // d p1
    ctas = sum_ctas(g1.N * 4);
    pool_adjoint_kernel<<<ctas, 256, 0, s>>>(g1, g2, 2, (const float4 *)u->gs1, (const float4 *)u->gup, (const float4 *)u->s1,
                                             (uint2 *)zn, colsum(E1B, ctas));
    next();
    if ((rc = conv_wgrad(u, E1B, u->a1, z, s))) return rc;
    if ((rc = conv_dgrad(u, E1B, z, masked(zn, u->a1), E1A, s))) return rc;
    next();
    if ((rc = conv_wgrad(u, E1A, u->x0, z, s))) return rc;
    sum_grads_kernel<<<(unsigned)(NLAYER + (u->sums.total + 31) / 32), 256, 0, s>>>(u->sums, u->wpart, u->bpart, u->grads);
    DST_CUDA_TRY(cudaGetLastError());
    return DST_OK;
}

// loss and gradients for input x (scaled by its norm) and target t (same scale)
static int loss_grad(dst_unet *u, const float *x, const float *t, cudaStream_t s) {
    const int64_t n = u->grid[0].N * u->C;
    int rc;
    if ((rc = set_input(u, x, t, s))) return rc;
    ConvOut o;
    o.f32 = u->y;
    if ((rc = forward(u, o, s))) return rc;
    const unsigned parts = sum_ctas(n / 4);
    u->sums.l[OUT].rows = (int)parts;
    loss_kernel<<<parts, 256, 0, s>>>(n / 4, log2i(u->C / 4), (int)parts, u->spart + SUM_CTAS, (const float4 *)u->y,
                                      t, u->scale, (uint2 *)u->z1, u->spart + 2 * SUM_CTAS,
                                      u->bpart + u->sums.l[OUT].bpart);
    loss_sum_kernel<<<1, 32, 0, s>>>((int)parts, u->spart + 2 * SUM_CTAS, u->dscr + 1);
    return backward(u, s);
}

// ---- preconditioner hook used by the solver --------------------------------------

int dst_internal_unet_correct(dst_unet *u, const dst_mesh *mesh, const float2 *rho, float2 *z, float2 *tmp,
                              cudaStream_t s, int *launches) {
    const int64_t nc = u->grid[0].N * u->C / 2;
    const float *x = reinterpret_cast<const float *>(rho);
    const float2 *y = reinterpret_cast<const float2 *>(u->y);
    *launches = (u->packed ? 0 : 1) + 2 + FORWARD_LAUNCHES + 1 + 2;
    int rc;
    if ((rc = set_input(u, x, nullptr, s))) return rc;
    ConvOut o;
    o.f32 = u->y;
    if ((rc = forward(u, o, s))) return rc;
    // the correction's scale for this input: alpha minimising ||rho - alpha A y||, so the
    // corrected direction never leaves a larger residual than the sweep alone
    if ((rc = dst_internal_apply(mesh, DST_FP32, y, tmp, s))) return rc;
    const int parts = (int)std::min<int64_t>(LS_PARTS, (nc + 2047) / 2048);
    ls_partials_kernel<<<parts, 256, 0, s>>>(nc, tmp, rho, u->part);
    ls_axpy_kernel<<<nblk(nc), 256, 0, s>>>(nc, parts, u->part, y, z);
    DST_CUDA_TRY(cudaGetLastError());
    return DST_OK;
}

bool dst_internal_unet_fits(const dst_unet *u, const dst_mesh *mesh) {
    return u && u->d == mesh->d && u->grid[0].N == mesh->nt * mesh->n_spatial && u->device == mesh->device;
}

// ---- C ABI ----------------------------------------------------------------------------

extern "C" int dst_unet_create(const dst_mesh *mesh, dst_unet **out) {
    if (!mesh || !out) return DST_ERR_ARG;
    *out = nullptr;
    if (mesh->nt > 0x7fffffff || mesh->n_spatial * mesh->nt > (1LL << 40)) return DST_ERR_ARG;
    return dst_internal_guard("dst_unet_create", [&] { return unet_create(mesh, out); });
}

extern "C" int dst_unet_destroy(dst_unet *u) {
    if (!u) return DST_OK;
    cudaFree(u->mem);
    delete u;
    return DST_OK;
}

extern "C" int dst_unet_num_params(const dst_unet *u, int64_t *n) {
    if (!u || !n) return DST_ERR_ARG;
    *n = u->nparams;
    return DST_OK;
}

extern "C" int dst_unet_set_params(dst_unet *u, const float *host) {
    if (!u || !host) return DST_ERR_ARG;
    DST_CUDA_TRY(cudaMemcpy(u->params, host, sizeof(float) * u->nparams, cudaMemcpyHostToDevice));
    DST_CUDA_TRY(cudaMemset(u->adam_m, 0, 2 * sizeof(float) * u->nparams));
    const float one = 1.0f;
    DST_CUDA_TRY(cudaMemcpy(u->gamma, &one, sizeof(float), cudaMemcpyHostToDevice));
    u->gamma_host = 1.0;
    u->packed = false;
    return DST_OK;
}

extern "C" int dst_unet_get_params(const dst_unet *u, float *host) {
    if (!u || !host) return DST_ERR_ARG;
    DST_CUDA_TRY(cudaMemcpy(host, u->params, sizeof(float) * u->nparams, cudaMemcpyDeviceToHost));
    return DST_OK;
}

extern "C" int dst_unet_forward(dst_unet *u, const void *x, void *y, void *stream) {
    if (!u || !x || !y) return DST_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int rc = set_input(u, (const float *)x, nullptr, s);
    if (rc) return rc;
    const bool aside = ((uintptr_t)y & 7) != 0;      // the last layer stores pairs of floats
    ConvOut o;                                       // y = gamma s U(x / s)
    o.f32 = aside ? u->y : (float *)y;
    o.s1 = u->gamma;
    o.s2 = u->scale;
    if (const int rf = forward(u, o, s)) return rf;
    if (aside)
        DST_CUDA_TRY(cudaMemcpyAsync(y, u->y, sizeof(float) * u->grid[0].N * u->C, cudaMemcpyDeviceToDevice, s));
    return DST_OK;
}

extern "C" int dst_unet_loss_grad(dst_unet *u, const void *x, const void *target, double *loss, float *grad_host,
                                  void *stream) {
    if (!u || !x || !target) return DST_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int rc = loss_grad(u, (const float *)x, (const float *)target, s);
    if (rc) return rc;
    if (loss) DST_CUDA_TRY(cudaMemcpyAsync(loss, u->dscr + 1, sizeof(double), cudaMemcpyDeviceToHost, s));
    if (grad_host)
        DST_CUDA_TRY(cudaMemcpyAsync(grad_host, u->grads, sizeof(float) * u->nparams, cudaMemcpyDeviceToHost, s));
    DST_CUDA_TRY(cudaStreamSynchronize(s));
    return DST_OK;
}

static int train(dst_unet *u, dst_mesh *mesh, int steps, float lr, uint64_t seed, float *loss_host, cudaStream_t s) {
    if (!dst_internal_unet_fits(u, mesh)) {
        dst_internal_set_error_detail("dst_unet_train: the network was created for another mesh");
        return DST_ERR_ARG;
    }
    SweepPlan plan;
    int rc = dst_sweep_plan(mesh, plan);
    if (rc) return rc;
    const int64_t n = mesh->n_unknowns;
    const size_t vb = (sizeof(float2) * (size_t)n + 255) & ~(size_t)255;
    const size_t sweep_bytes = dst_sweep_scratch_bytes(plan, n);
    char *scr = nullptr;
    if (cudaMallocAsync((void **)&scr, 5 * vb + sweep_bytes + 256, s) != cudaSuccess) {
        cudaGetLastError();
        return DST_ERR_OOM;
    }
    float2 *e = (float2 *)scr, *r = (float2 *)(scr + vb), *z = (float2 *)(scr + 2 * vb), *az = (float2 *)(scr + 3 * vb),
           *tg = (float2 *)(scr + 4 * vb);
    double *lossd = nullptr;
    rc = dst_sweep_setup(mesh, plan, scr + 5 * vb, s);
    std::vector<double> losses(steps > 0 ? steps : 1);
    if (rc == DST_OK && cudaMallocAsync((void **)&lossd, sizeof(double) * (steps > 0 ? steps : 1), s) != cudaSuccess) {
        cudaGetLastError();
        rc = DST_ERR_OOM;
    }
    const float b1 = 0.9f, b2 = 0.999f;
    for (int it = 0; it < steps && rc == DST_OK; ++it) {
        // a training pair from the method: e random, r = A e, z = M_CN r, rho = r - A z, target e - z
        randn_kernel<<<nblk(n), 256, 0, s>>>(n, seed + (uint64_t)it * 0x9E3779B97F4A7C15ull, e);
        if ((rc = dst_internal_apply(mesh, DST_FP32, e, r, s))) break;
        if ((rc = dst_sweep_apply(plan, n, r, z, s))) break;
        if ((rc = dst_internal_apply(mesh, DST_FP32, z, az, s))) break;
        if ((rc = dst_k_sub_f32(n, r, az, r, s))) break;                  // r <- rho
        if ((rc = dst_k_sub_f32(n, e, z, tg, s))) break;                  // target
        if ((rc = loss_grad(u, (const float *)r, (const float *)tg, s))) break;
        if (cudaMemcpyAsync(lossd + it, u->dscr + 1, sizeof(double), cudaMemcpyDeviceToDevice, s) != cudaSuccess) {
            rc = DST_ERR_CUDA;
            break;
        }
        const float c1 = 1.f - std::pow(b1, (float)(it + 1)), c2 = 1.f - std::pow(b2, (float)(it + 1));
        adam_kernel<<<nblk(u->nparams), 256, 0, s>>>(u->nparams, u->params, u->grads, u->adam_m, u->adam_v, lr, b1, b2,
                                                      c1, c2, 1e-8f);
        if ((rc = pack(u, s))) break;
    }
    // output scale: the least-squares factor gamma = <U, t> / ||U||^2 over fresh pairs, so
    // that the scaled correction's error on them is never above the sweep's own
    if (rc == DST_OK && steps > 0) {
        const int nval = 8;
        double *acc = u->dscr + 2;                      // [2], [3]; dscr[2] is reused by loss_grad only
        if (cudaMemsetAsync(acc, 0, 2 * sizeof(double), s) != cudaSuccess) rc = DST_ERR_CUDA;
        for (int it = 0; it < nval && rc == DST_OK; ++it) {
            randn_kernel<<<nblk(n), 256, 0, s>>>(n, ~seed + (uint64_t)it * 0xD1B54A32D192ED03ull, e);
            if ((rc = dst_internal_apply(mesh, DST_FP32, e, r, s))) break;
            if ((rc = dst_sweep_apply(plan, n, r, z, s))) break;
            if ((rc = dst_internal_apply(mesh, DST_FP32, z, az, s))) break;
            if ((rc = dst_k_sub_f32(n, r, az, r, s))) break;
            if ((rc = dst_k_sub_f32(n, e, z, tg, s))) break;
            if ((rc = set_input(u, (const float *)r, nullptr, s))) break;
            ConvOut o;
            o.f32 = u->y;
            if ((rc = forward(u, o, s))) break;
            dot_kernel<<<1, 256, 0, s>>>(2 * n, u->y, (const float *)tg, u->scale, acc);
        }
        double hacc[2] = {0.0, 0.0};
        if (rc == DST_OK && (cudaMemcpyAsync(hacc, acc, sizeof(hacc), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                             cudaStreamSynchronize(s) != cudaSuccess))
            rc = DST_ERR_CUDA;
        if (rc == DST_OK) {
            double gmm = hacc[1] > 0.0 ? hacc[0] / hacc[1] : 0.0;
            if (!(gmm > 0.0)) gmm = 0.0;
            const float gf = (float)gmm;
            u->gamma_host = gmm;
            if (cudaMemcpyAsync(u->gamma, &gf, sizeof(float), cudaMemcpyHostToDevice, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess)
                rc = DST_ERR_CUDA;
        }
    }
    if (rc == DST_OK && steps > 0 && loss_host) {
        if (cudaMemcpyAsync(losses.data(), lossd, sizeof(double) * steps, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            rc = DST_ERR_CUDA;
        for (int i = 0; i < steps; ++i) loss_host[i] = (float)losses[i];
    }
    if (lossd) cudaFreeAsync(lossd, s);
    cudaFreeAsync(scr, s);
    if (rc == DST_OK) DST_CUDA_TRY(cudaStreamSynchronize(s));
    return rc;
}

extern "C" int dst_unet_train(dst_unet *u, dst_mesh *mesh, int steps, float lr, uint64_t seed, float *loss_host,
                              void *stream) {
    if (!u || !mesh || steps < 0 || !(lr > 0)) return DST_ERR_ARG;
    return dst_internal_guard("dst_unet_train", [&] { return train(u, mesh, steps, lr, seed, loss_host, (cudaStream_t)stream); });
}

extern "C" int dst_unet_output_scale(const dst_unet *u, double *gamma) {
    if (!u || !gamma) return DST_ERR_ARG;
    *gamma = u->gamma_host;
    return DST_OK;
}

extern "C" int dst_set_learned_precond(dst_mesh *mesh, dst_unet *u) {
    if (!mesh) return DST_ERR_ARG;
    if (u && !dst_internal_unet_fits(u, mesh)) {
        dst_internal_set_error_detail("dst_set_learned_precond: the network was created for another mesh");
        return DST_ERR_ARG;
    }
    mesh->unet = u;
    return DST_OK;
}
