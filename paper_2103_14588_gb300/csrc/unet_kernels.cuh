// Kernels of the convolutional U-Net preconditioner: implicit-GEMM convolutions
// on BF16 tensor cores with FP32 accumulation (mma.sync m16n8k16), and the
// element-wise pieces (pooling, the adjoints of pooling and upsampling).
//
// Activations are arrays [node][channel] over a D-dimensional node grid
// (t slowest, then z, y, x; only the axes the mesh has).  What a convolution reads is
// stored in BF16, rounded once by its producer; what is added or pooled in FP32 stays
// FP32.  A convolution with kernel 3 in every axis (taps = 3^D, zero padding that keeps
// the size) or kernel 1 (one tap) is the cross-correlation
// out[n][co] = b[co] + sum_tap sum_ci in[n + off(tap)][ci] W[co][ci][tap],
// evaluated as a GEMM with M = nodes, N = output channels and K = taps x input
// channels; K index k = tap * Ci + ci, tap in row-major order of the kernel
// offsets (-1, 0, 1) per axis, 16 of them per tensor-core instruction in that order.
//
// The layers are small (16 to 64 channels, 6 GFLOP in all on a 48^3 grid), so the
// tensor cores are never the limit: what is, is the instructions around them and the
// launches, and on the coarse grids the latency of a chain of taps that few warps walk.
// So a thread works out its rows' coordinates once; a tap is then a node offset and a mask
// of the axis ends it must not start from (a table in shared memory).  Taps stream through
// a shared-memory ring (cp.async, zero-filled outside the grid) a few stages ahead of the
// products; weights are packed in fragment order.
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

namespace dst_nn {

typedef __nv_bfloat16 bf16;

struct UGrid {
    int D;            // axes (2, 3 or 4)
    int n[4];         // nodes per axis, slowest first
    int64_t N;        // nodes (below 2^31: 200 bytes of activations each)
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ uint2 pack_bf16x4(float4 v) { return make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w)); }
// whether the low / high BF16 of a pair is above zero
__device__ __forceinline__ bool pos_lo(uint32_t v) { return __uint_as_float(v << 16) > 0.f; }
__device__ __forceinline__ bool pos_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u) > 0.f; }

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// coordinates of node r (slowest axis first)
__device__ __forceinline__ void coords(const UGrid &g, unsigned r, int (&c)[4]) {
#pragma unroll
    for (int a = 3; a >= 0; --a)
        if (a < g.D) {
            const unsigned q = r / (unsigned)g.n[a];
            c[a] = (int)(r - q * (unsigned)g.n[a]);
            r = q;
        }
}
// node of the coarse grid above a fine node's coordinates
__device__ __forceinline__ unsigned parent(const UGrid &c, const int (&x)[4]) {
    unsigned q = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a)
        if (a < c.D) q = q * (unsigned)c.n[a] + (unsigned)(x[a] >> 1);
    return q;
}

struct ConvArgs {
    UGrid g;
    UGrid up;                       // grid of `in` when rows read their parent node (coarse != 0)
    int coarse;
    int lci, taps, chunks;          // log2 of the input channels, kernel taps, K / 16
    int co, ntiles;                 // output channels stored, output channels / 8 rounded up
    const bf16 *in;                 // [N][ci]
    const bf16 *zeros;              // 64 channels of zeros
    const uint32_t *w;              // fragments [chunk][ntile][lane][2]
    const float *bias;              // [co] or null
    const float *res;               // [N][co] added before the activation, or null
    int relu;
    const bf16 *mask;               // [N][co]: 0 where not above zero, or null
    const float *s1, *s2;           // device scalars: the stored value is *s1 * *s2 * v, or null
    float *out32;                   // [N][co] or null
    bf16 *out16;                    // [N][co] or null
    float *colsum;                  // [gridDim.x][co] sums over the CTA's nodes, or null
};

struct Tap {
    long long off;                  // offset in elements of `in`
    int ends;                       // axis ends (bit 2a: first node, 2a + 1: last) it must not start from
    int pad;
};

constexpr int CONV_WARPS = 4;
constexpr int CONV_STAGES = 4;

__device__ __forceinline__ void copy_or_zero16(void *dst, const void *src, bool ok) {
    const int n = ok ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(n) : "memory");
}
__device__ __forceinline__ void copy_or_zero8(void *dst, const void *src, bool ok) {
    const int n = ok ? 8 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(n) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// Shared memory of the ring.  A stage holds the rows of one offset of the slower axes, with
// a row on each side, and the weights of its three taps: the taps along x read the same
// rows, shifted by one (at an end of the x line a row of zeros).  Eight rows of any 16-byte
// column lie on different banks (the column is swizzled by the row).
template <int NT, int MT, int CI16>
struct ConvShape {
    static constexpr int ROWS = 16 * MT * CONV_WARPS + 2, COLS = 2 * CI16;
    static constexpr int A = ROWS * CI16 * 32, B_TAP = CI16 * NT * 256;
    static constexpr int STAGE = A + 3 * B_TAP;
    static constexpr size_t SMEM = (size_t)CONV_STAGES * STAGE + CI16 * 32;
    __device__ static int at(int row, int col) {
        const int sw = CI16 == 1 ? (row >> 2) & 1 : CI16 == 2 ? (row >> 1) & 3 : row & 7;
        return (row * COLS + (col ^ sw)) * 16;
    }
};

// One warp: 16 MT consecutive nodes x 8 NT output channels (blockIdx.y: which).  CI16: input
// channels / 16; 0 (any number) without the ring.
// 16 -> 16 channels at 48^3 (1.5 GFLOP): 19 us with loads through L1, 15 us staged; 64 -> 64
// channels at 12^3: 58 and 12 us (253 and 388 us with divisions per fragment).
template <int NT, int MT, int CI16>
__global__ void __launch_bounds__(32 * CONV_WARPS) conv_kernel(ConvArgs a) {
    extern __shared__ __align__(16) unsigned char ring[];
    __shared__ Tap tab[82];
    __shared__ float cs[CONV_WARPS][NT * 8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, tg = lane & 3;
    const int ci = 1 << a.lci;
    // staged: the offsets of the slower axes; else every tap, the one after the last (K
    // padded to a multiple of 16) starting from nowhere
    constexpr int xt = CI16 > 0 ? 3 : 1;                   // (a staged convolution has kernel 3)
    const int entries = a.taps / xt;
    for (int t = threadIdx.x; t <= entries; t += blockDim.x) {
        Tap e{0, t < entries ? 0 : 1 << 8, 0};
        if (a.taps > 1 && t < entries) {
            int rest = xt == 3 ? 3 * t + 1 : t;
            long long stride = 1;
            for (int ax = a.g.D - 1; ax >= 0; --ax) {
                const int o = rest % 3 - 1;
                rest /= 3;
                e.off += o * stride;
                stride *= a.g.n[ax];
                if (o < 0) e.ends |= 1 << (2 * ax);
                if (o > 0) e.ends |= 2 << (2 * ax);
            }
            e.off *= ci;
        }
        tab[t] = e;
    }
    // a row's first channel and the axis ends it lies on; a row outside the grid reads nothing
    auto place = [&](int64_t r, const bf16 *&at, int &ends) {
        at = a.in;
        ends = -1;
        if (r < 0 || r >= a.g.N) return;
        int c[4];
        int e = 1 << 8;
        coords(a.g, (unsigned)r, c);
#pragma unroll
        for (int ax = 0; ax < 4; ++ax)
            if (ax < a.g.D) e |= (c[ax] == 0 ? 1 << (2 * ax) : 0) | (c[ax] == a.g.n[ax] - 1 ? 2 << (2 * ax) : 0);
        ends = e;
        at = a.in + ((a.coarse ? (int64_t)parent(a.up, c) : r) << a.lci);
    };
    const int64_t cta0 = (int64_t)blockIdx.x * (16 * MT * CONV_WARPS), m0 = cta0 + warp * (16 * MT);
    float acc[MT][NT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
    const size_t wstep = (size_t)a.ntiles * 32;
    if constexpr (CI16 > 0) {
        using S = ConvShape<NT, MT, CI16>;
        constexpr int THREADS = 32 * CONV_WARPS, MINE = (S::ROWS * S::COLS + THREADS - 1) / THREADS;   // copies per thread
        const bf16 *src[MINE];
        int ends[MINE], dst[MINE];
#pragma unroll
        for (int i = 0; i < MINE; ++i) {
            const int k = threadIdx.x + i * THREADS, row = k / S::COLS, col = k % S::COLS;
            src[i] = a.in;
            ends[i] = -1;
            if (row < S::ROWS) place(cta0 - 1 + row, src[i], ends[i]);
            src[i] += col * 8;
            dst[i] = row < S::ROWS ? S::at(row, col) : -1;
        }
        // the x ends of the rows this lane addresses
        int xe[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const bf16 *q;
            int e;
            place(m0 + m * 16 + (lane & 15), q, e);
            xe[m] = (e >> (2 * (a.g.D - 1))) & 3;
        }
        unsigned char *zero_row = ring + CONV_STAGES * S::STAGE;
        if (threadIdx.x < S::COLS) reinterpret_cast<uint4 *>(zero_row)[threadIdx.x] = make_uint4(0, 0, 0, 0);
        __syncthreads();
        const uint4 *wsrc = reinterpret_cast<const uint4 *>(reinterpret_cast<const uint2 *>(a.w) + (size_t)blockIdx.y * NT * 32);
        auto issue = [&](int st) {
            if (st < entries) {
                unsigned char *base = ring + (st % CONV_STAGES) * S::STAGE;
                const Tap t = tab[st];
#pragma unroll
                for (int i = 0; i < MINE; ++i) {
                    const bool ok = ends[i] != -1 && !(ends[i] & t.ends);
                    if (dst[i] >= 0) copy_or_zero16(base + dst[i], src[i] + (ok ? t.off : 0), ok);
                }
                for (int i = threadIdx.x; i < xt * S::B_TAP / 16; i += THREADS) {
                    const int c = i / (NT * 16), o = i % (NT * 16);            // chunk of the stage's taps
                    copy_or_zero16(base + S::A + i * 16, wsrc + ((size_t)(st * xt * CI16 + c) * wstep) / 2 + o, true);
                }
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        };
        for (int st = 0; st < CONV_STAGES - 1; ++st) issue(st);
        for (int st = 0; st < entries; ++st) {
            asm volatile("cp.async.wait_group %0;\n" ::"n"(CONV_STAGES - 2) : "memory");
            __syncthreads();
            issue(st + CONV_STAGES - 1);
            const unsigned char *base = ring + (st % CONV_STAGES) * S::STAGE;
            const uint2 *wd = reinterpret_cast<const uint2 *>(base + S::A) + lane;
            auto tap = [&](int dx, int u) {                // dx: -1, 0, 1; u: place among the stage's weights
#pragma unroll
                for (int c = 0; c < CI16; ++c) {
                    uint32_t af[MT][4];
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        const bool out = (dx < 0 && (xe[m] & 1)) || (dx > 0 && (xe[m] & 2));
                        ldsm4(af[m], out ? zero_row
                                         : base + S::at(warp * (16 * MT) + m * 16 + (lane & 15) + 1 + dx, 2 * c + (lane >> 4)));
                    }
#pragma unroll
                    for (int j = 0; j < NT; ++j) {
                        const uint2 b = wd[((u * CI16 + c) * NT + j) * 32];
#pragma unroll
                        for (int m = 0; m < MT; ++m) mma_16816(acc[m][j], af[m], b.x, b.y);
                    }
                }
            };
            tap(-1, 0);
            tap(0, 1);
            tap(1, 2);
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    } else {
        __syncthreads();
        // four or eight input channels (a chunk spans several taps) or one tap: through L1
        const bf16 *row[MT][2];
        int ends[MT][2];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) place(m0 + m * 16 + h * 8 + g, row[m][h], ends[m][h]);
        const uint2 *w = reinterpret_cast<const uint2 *>(a.w) + ((size_t)blockIdx.y * NT) * 32 + lane;
#pragma unroll 4
        for (int kc = 0; kc < a.chunks; ++kc) {
            uint32_t af[MT][4];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int k = kc * 16 + half * 8 + 2 * tg;
                const Tap t = tab[min(k >> a.lci, a.taps)];
                const int ch = k & (ci - 1);
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const bf16 *q = (ends[m][h] & t.ends) ? a.zeros : row[m][h] + (t.off + ch);
                        af[m][2 * half + h] = __ldg(reinterpret_cast<const uint32_t *>(q));
                    }
            }
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const uint2 b = __ldg(w + kc * wstep + j * 32);
#pragma unroll
                for (int m = 0; m < MT; ++m) mma_16816(acc[m][j], af[m], b.x, b.y);
            }
        }
    }
    const float scale = a.s1 ? *a.s1 * *a.s2 : 1.f;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int cc = (blockIdx.y * NT + j) * 8 + 2 * tg;
        float sum0 = 0.f, sum1 = 0.f;
        if (cc < a.co) {                                  // co is even
            const float b0 = a.bias ? a.bias[cc] : 0.f, b1 = a.bias ? a.bias[cc + 1] : 0.f;
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int64_t r = m0 + m * 16 + h * 8 + g;
                    if (r >= a.g.N) continue;
                    const int64_t at = r * a.co + cc;
                    float v0 = acc[m][j][2 * h], v1 = acc[m][j][2 * h + 1];
                    if (a.bias) { v0 += b0; v1 += b1; }
                    if (a.res) {
                        const float2 q = *reinterpret_cast<const float2 *>(a.res + at);
                        v0 += q.x; v1 += q.y;
                    }
                    if (a.relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); }
                    if (a.mask) {
                        const uint32_t y = *reinterpret_cast<const uint32_t *>(a.mask + at);
                        v0 = pos_lo(y) ? v0 : 0.f;
                        v1 = pos_hi(y) ? v1 : 0.f;
                    }
                    if (a.s1) { v0 = scale * v0; v1 = scale * v1; }
                    if (a.out32) *reinterpret_cast<float2 *>(a.out32 + at) = make_float2(v0, v1);
                    if (a.out16) *reinterpret_cast<uint32_t *>(a.out16 + at) = pack_bf16(v0, v1);
                    sum0 += v0; sum1 += v1;
                }
        }
        if (a.colsum) {
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                sum0 += __shfl_xor_sync(0xffffffffu, sum0, o);
                sum1 += __shfl_xor_sync(0xffffffffu, sum1, o);
            }
            if (g == 0) { cs[warp][j * 8 + 2 * tg] = sum0; cs[warp][j * 8 + 2 * tg + 1] = sum1; }
        }
    }
    if (a.colsum) {
        __syncthreads();
        const int cc = blockIdx.y * NT * 8 + threadIdx.x;
        if (threadIdx.x < NT * 8 && cc < a.co) {
            float t = 0.f;
#pragma unroll
            for (int q = 0; q < CONV_WARPS; ++q) t += cs[q][threadIdx.x];
            a.colsum[(size_t)blockIdx.x * a.co + cc] = t;
        }
    }
}

// ---- weight gradients -------------------------------------------------------
//
// dW[co][k] = sum_n dz[n][co] in[n + off(tap(k))][ci(k)]: a GEMM with M = co, N = k and
// K = nodes, both operands transposed on their way from shared memory (ldmatrix.trans).
// Kernel 3: a CTA walks segments of x lines; each warp stages the neighbour line of one
// offset of the slower axes (with a node on each side, zeros outside the grid) and owns
// its three taps, so a staged node serves three taps and a line's dz serves every warp.
// The CTA's sum over its segments goes to its own slice of dw; the slices are summed in
// order afterwards, so that training is reproducible.
struct WgradArgs {
    UGrid g;
    UGrid up;               // kernel 1: grid of `in` when rows read their parent node (coarse != 0)
    int coarse;
    int ci, taps, kpad, co;
    const bf16 *in;         // layer input [N][ci]
    const bf16 *dz;         // gradient of the layer's output before its activation [N][co]
    float *dw;              // [slices][co][kpad]
    int seg, segs, items;   // nodes per segment, segments per line, segments in all
    int per_cta;
};

__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"((unsigned)__cvta_generic_to_shared(p)));
}
__device__ __forceinline__ void ldsm2t(uint32_t &a, uint32_t &b, const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(a), "=r"(b) : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// Row pitch in shared memory: the channels and 16 bytes, so that the eight rows of a
// transposing load fall on different banks.
__host__ __device__ constexpr int wg_pitch(int channels) { return channels * 2 + 16; }
constexpr int WG_DZ = wg_pitch(16);            // dz: 16 channels of the CTA's row block

constexpr int WG_MAX_SEG = 64;                 // nodes of a segment of an x line, at most
__host__ __device__ inline int wg_padded(int seg) { return (seg + 15) / 16 * 16; }
__host__ __device__ inline size_t wg_buffer(int ci8, int warps, int seg) {
    return (size_t)warps * (wg_padded(seg) + 2) * wg_pitch(ci8 * 8) + (size_t)wg_padded(seg) * WG_DZ;
}

// CI8: input channels / 8 (at least 1).  blockIdx = (slice, 16 co, group of offsets).
template <int CI8>
__global__ void __launch_bounds__(288) wgrad3_kernel(WgradArgs a) {
    extern __shared__ __align__(16) unsigned char wsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int g = lane >> 2, tg = lane & 3;
    constexpr int P = wg_pitch(CI8 * 8);
    const int segp = wg_padded(a.seg), nx = a.g.n[a.g.D - 1];
    const size_t bufb = wg_buffer(CI8, warps, a.seg);
    const int q = blockIdx.z * warps + warp;               // offset of the slower axes, row-major
    const int co0 = blockIdx.y * 16;
    // a mesh of two components has four input channels: the upper half of a row stays zero
    if (a.ci < 8) {
        for (size_t i = threadIdx.x; i < 2 * bufb / 16; i += blockDim.x) reinterpret_cast<uint4 *>(wsm)[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
    }
    float acc[3][CI8][4];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int j = 0; j < CI8; ++j) acc[d][j][0] = acc[d][j][1] = acc[d][j][2] = acc[d][j][3] = 0.f;
    const int first = blockIdx.x * a.per_cta, last = min(first + a.per_cta, a.items);
    auto stage = [&](int item, int buf) {
        if (item < last) {
            unsigned char *base = wsm + buf * bufb, *line = base + (size_t)warp * (segp + 2) * P,
                          *dzt = base + (size_t)warps * (segp + 2) * P;
            const int l = item / a.segs, x0 = (item - l * a.segs) * a.seg, len = min(a.seg, nx - x0);
            // the line at this warp's offset
            int rest = l, off = q;
            int64_t nb = 0, stride = 1;
            bool ok = true;
            for (int ax = a.g.D - 2; ax >= 0; --ax) {
                const int c = rest % a.g.n[ax] + off % 3 - 1;
                rest /= a.g.n[ax];
                off /= 3;
                ok = ok && c >= 0 && c < a.g.n[ax];
                nb += c * stride;
                stride *= a.g.n[ax];
            }
            const bf16 *src = a.in + (ok ? (nb * nx) * a.ci : 0);
            if (a.ci >= 8) {
                for (int i = lane; i < (segp + 2) * CI8; i += 32) {
                    const int r = i / CI8, ch = i % CI8, x = x0 - 1 + r;
                    const bool in = ok && x >= 0 && x < nx && r < len + 2;
                    copy_or_zero16(line + r * P + ch * 16, src + (in ? (int64_t)x * a.ci + ch * 8 : 0), in);
                }
            } else {
                for (int r = lane; r < segp + 2; r += 32) {
                    const int x = x0 - 1 + r;
                    const bool in = ok && x >= 0 && x < nx && r < len + 2;
                    copy_or_zero8(line + r * P, src + (in ? (int64_t)x * a.ci : 0), in);
                }
            }
            const bf16 *dsrc = a.dz + ((int64_t)l * nx + x0) * a.co + co0;
            for (int i = threadIdx.x; i < segp * 2; i += blockDim.x) {
                const int r = i >> 1, ch = i & 1;
                copy_or_zero16(dzt + r * WG_DZ + ch * 16, dsrc + (r < len ? (int64_t)r * a.co + ch * 8 : 0), r < len);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    stage(first, 0);
    for (int item = first; item < last; ++item) {
        const int buf = (item - first) & 1;
        stage(item + 1, buf ^ 1);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();
        const unsigned char *base = wsm + buf * bufb, *line = base + (size_t)warp * (segp + 2) * P,
                            *dzt = base + (size_t)warps * (segp + 2) * P;
        for (int k0 = 0; k0 < segp; k0 += 16) {
            uint32_t af[4];
            ldsm4t(af, dzt + (k0 + (lane & 7) + ((lane >> 4) << 3)) * WG_DZ + ((lane >> 3) & 1) * 16);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const unsigned char *rows = line + (k0 + d + (lane & 15)) * P;
                if (CI8 == 1) {
                    uint32_t b0, b1;
                    ldsm2t(b0, b1, rows);
                    mma_16816(acc[d][0], af, b0, b1);
                } else {
#pragma unroll
                    for (int j = 0; j < CI8; j += 2) {
                        uint32_t b[4];
                        ldsm4t(b, rows + (j + (lane >> 4)) * 16);
                        mma_16816(acc[d][j], af, b[0], b[1]);
                        mma_16816(acc[d][j + 1 < CI8 ? j + 1 : 0], af, b[2], b[3]);
                    }
                }
            }
        }
        __syncthreads();
    }
    float *part = a.dw + (size_t)blockIdx.x * a.co * a.kpad;
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int j = 0; j < CI8; ++j) {
            const int ch = j * 8 + 2 * tg, k = (q * 3 + d) * a.ci + ch;
            if (ch < a.ci) {
                *reinterpret_cast<float2 *>(part + (size_t)(co0 + g) * a.kpad + k) = make_float2(acc[d][j][0], acc[d][j][1]);
                *reinterpret_cast<float2 *>(part + (size_t)(co0 + g + 8) * a.kpad + k) = make_float2(acc[d][j][2], acc[d][j][3]);
            }
        }
}

// Kernel 1: each warp of the CTA sums its own nodes, 32 at a time, into its own slice.
template <int CI8>
__global__ void __launch_bounds__(128) wgrad1_kernel(WgradArgs a) {
    constexpr int P = wg_pitch(CI8 * 8), ROWS = 32;
    __shared__ __align__(16) unsigned char sm[4][2][ROWS * (P + WG_DZ)];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, tg = lane & 3, co0 = blockIdx.y * 16;
    for (int i = threadIdx.x; i < (int)sizeof(sm) / 16; i += blockDim.x) reinterpret_cast<uint4 *>(sm)[i] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    float acc[CI8][4];
#pragma unroll
    for (int j = 0; j < CI8; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    const int slice = blockIdx.x * 4 + warp;
    const int first = min(slice * a.per_cta, a.items), last = min(first + a.per_cta, a.items);
    auto stage = [&](int item, int buf) {
        if (item < last) {
            unsigned char *in = sm[warp][buf], *dzt = in + ROWS * P;
            const int64_t r = (int64_t)item * ROWS + lane;           // one row per lane
            const bool ok = r < a.g.N;
            int64_t from = ok ? r : 0;
            if (a.coarse && ok) {
                int c[4];
                coords(a.g, (unsigned)r, c);
                from = parent(a.up, c);
            }
#pragma unroll
            for (int ch = 0; ch < CI8; ++ch) copy_or_zero16(in + lane * P + ch * 16, a.in + from * a.ci + ch * 8, ok);
            if (a.co < 8) copy_or_zero8(dzt + lane * WG_DZ, a.dz + (ok ? r : 0) * a.co, ok);
            else
                for (int ch = 0; ch < 2; ++ch)
                    copy_or_zero16(dzt + lane * WG_DZ + ch * 16, a.dz + (ok ? r : 0) * a.co + co0 + ch * 8,
                                   ok && co0 + ch * 8 < a.co);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    stage(first, 0);
    for (int item = first; item < last; ++item) {
        const int buf = (item - first) & 1;
        stage(item + 1, buf ^ 1);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncwarp();
        const unsigned char *in = sm[warp][buf], *dzt = in + ROWS * P;
#pragma unroll
        for (int k0 = 0; k0 < ROWS; k0 += 16) {
            uint32_t af[4];
            ldsm4t(af, dzt + (k0 + (lane & 7) + ((lane >> 4) << 3)) * WG_DZ + ((lane >> 3) & 1) * 16);
#pragma unroll
            for (int j = 0; j < CI8; j += 2) {
                uint32_t b[4];
                ldsm4t(b, in + (k0 + (lane & 15)) * P + (j + (lane >> 4)) * 16);
                mma_16816(acc[j], af, b[0], b[1]);
                mma_16816(acc[j + 1], af, b[2], b[3]);
            }
        }
        __syncwarp();
    }
    float *part = a.dw + (size_t)slice * a.co * a.kpad;
#pragma unroll
    for (int j = 0; j < CI8; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (co0 + g + 8 * h < a.co)
                *reinterpret_cast<float2 *>(part + (size_t)(co0 + g + 8 * h) * a.kpad + j * 8 + 2 * tg) =
                    make_float2(acc[j][2 * h], acc[j][2 * h + 1]);
}

// Where one layer's partial sums lie and where its gradients go.
struct GradLayer {
    int co, ci, taps, kpad, slices, rows;
    int64_t woff, boff;             // in the flat gradient
    int64_t wpart, bpart;           // in the partial buffers
    int64_t first;                  // first (co, k) of the layer among all layers'
};
struct GradLayers {
    int n, bias_ctas;
    int64_t total;                  // (co, k) pairs of all layers
    GradLayer l[11];
};

// The flat gradient: every weight the sum of its slices in order; one CTA per layer (the
// first ones) sums the rows of the bias gradients.
__global__ void __launch_bounds__(256) sum_grads_kernel(GradLayers L, const float *__restrict__ wpart,
                                                        const float *__restrict__ bpart, float *__restrict__ grad) {
    if ((int)blockIdx.x < L.n) {
        __shared__ float red[256];
        const GradLayer &l = L.l[blockIdx.x];
        const int per = 256 / l.co * l.co, c = threadIdx.x % l.co;
        float t = 0.f;
        if ((int)threadIdx.x < per) {
            const float *p = bpart + l.bpart;
#pragma unroll 8
            for (int64_t i = threadIdx.x; i < (int64_t)l.rows * l.co; i += per) t += p[i];
        }
        red[threadIdx.x] = t;
        __syncthreads();
        if ((int)threadIdx.x < l.co) {
            t = 0.f;
            for (int i = c; i < per; i += l.co) t += red[i];
            grad[l.boff + c] = t;
        }
        return;
    }
    // 32 pairs per CTA, their slices over eight warps
    __shared__ float part[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)(blockIdx.x - L.n) * 32 + lane;
    int k = 0;
    while (k + 1 < L.n && i >= L.l[k + 1].first) ++k;
    const GradLayer &l = L.l[k];
    const int at = (int)(i - l.first), o = at / l.kpad, kk = at - o * l.kpad;
    const bool live = i < L.total && kk < l.taps * l.ci;
    float t = 0.f;
    if (live) {
        const float *p = wpart + l.wpart + at;
        const int64_t step = (int64_t)l.co * l.kpad;
#pragma unroll 4
        for (int s = warp; s < l.slices; s += 8) t += p[s * step];
    }
    part[warp][lane] = t;
    __syncthreads();
    if (warp == 0 && live) {
        for (int w = 1; w < 8; ++w) t += part[w][lane];
        grad[l.woff + ((int64_t)o * l.ci + kk % l.ci) * l.taps + kk / l.ci] = t;
    }
}

// ---- element-wise pieces, four channels per thread ----------------------------

// Sum of four channels over the 2^D fine nodes of a coarse node (nodes past an odd end
// count as zero), in order; the loads of eight nodes in flight together.
__device__ __forceinline__ float4 fine_sum(const UGrid &f, const int (&cc)[4], int lq, int k, const float4 *__restrict__ in) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int m0 = 0; m0 < 1 << f.D; m0 += 8) {
        float4 v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int m = m0 + e;
            int64_t r = 0;
            bool ok = m < 1 << f.D;
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (a < f.D) {
                    const int x = 2 * cc[a] + ((m >> (f.D - 1 - a)) & 1);
                    ok = ok && x < f.n[a];
                    r = r * f.n[a] + x;
                }
            v[e] = ok ? __ldg(in + (r << lq) + k) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) { s.x += v[e].x; s.y += v[e].y; s.z += v[e].z; s.w += v[e].w; }
    }
    return s;
}

// out[q] = mean of in over the fine nodes of q
__global__ void __launch_bounds__(256) pool_kernel(UGrid f, UGrid c, int lq, const float4 *__restrict__ in, uint2 *__restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;       // (node, four channels)
    if (i >= c.N << lq) return;
    int cc[4];
    coords(c, (unsigned)(i >> lq), cc);
    const float4 s = fine_sum(f, cc, lq, (int)(i & ((1 << lq) - 1)), in);
    const float w = 1.f / (float)(1 << f.D);               // a power of two
    out[i] = pack_bf16x4(make_float4(s.x * w, s.y * w, s.z * w, s.w * w));
}

// Column sums of a CTA's nodes: every thread keeps the same four channels throughout.
__device__ __forceinline__ void cta_colsum(float4 t, int lq, float *colsum) {
    __shared__ float4 red[256];
    red[threadIdx.x] = t;
    __syncthreads();
    const int nq = 1 << lq;
    if ((int)threadIdx.x < nq) {
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = threadIdx.x; i < 256; i += nq) { s.x += red[i].x; s.y += red[i].y; s.z += red[i].z; s.w += red[i].w; }
        reinterpret_cast<float4 *>(colsum)[((int64_t)blockIdx.x << lq) + threadIdx.x] = s;
    }
}

// dz[q] = (y[q] > 0) sum of d over the fine nodes of q (the adjoint of the upsampling)
__global__ void __launch_bounds__(256) up_adjoint_kernel(UGrid f, UGrid c, int lq, const float4 *__restrict__ d,
                                                         const uint2 *__restrict__ y, uint2 *__restrict__ dz,
                                                         float *__restrict__ colsum) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < c.N << lq; i += (int64_t)gridDim.x * 256) {
        int cc[4];
        coords(c, (unsigned)(i >> lq), cc);
        float4 s = fine_sum(f, cc, lq, (int)(i & ((1 << lq) - 1)), d);
        const uint2 m = y[i];
        s = make_float4(pos_lo(m.x) ? s.x : 0.f, pos_hi(m.x) ? s.y : 0.f, pos_lo(m.y) ? s.z : 0.f, pos_hi(m.y) ? s.w : 0.f);
        dz[i] = pack_bf16x4(s);
        t.x += s.x; t.y += s.y; t.z += s.z; t.w += s.w;
    }
    cta_colsum(t, lq, colsum);
}

// dz[p] = (y[p] > 0) (d[p] + dc[p / 2] / 2^D) (the adjoint of the pooling added to d)
__global__ void __launch_bounds__(256) pool_adjoint_kernel(UGrid f, UGrid c, int lq, const float4 *__restrict__ d,
                                                           const float4 *__restrict__ dc, const float4 *__restrict__ y,
                                                           uint2 *__restrict__ dz, float *__restrict__ colsum) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    const float w = 1.f / (float)(1 << f.D);
    for (int64_t i = blockIdx.x * 256LL + threadIdx.x; i < f.N << lq; i += (int64_t)gridDim.x * 256) {
        int cc[4];
        coords(f, (unsigned)(i >> lq), cc);
        const float4 u = d[i], v = __ldg(dc + ((int64_t)parent(c, cc) << lq) + (i & ((1 << lq) - 1))), m = y[i];
        const float4 s = make_float4(m.x > 0.f ? u.x + v.x * w : 0.f, m.y > 0.f ? u.y + v.y * w : 0.f,
                                     m.z > 0.f ? u.z + v.z * w : 0.f, m.w > 0.f ? u.w + v.w * w : 0.f);
        dz[i] = pack_bf16x4(s);
        t.x += s.x; t.y += s.y; t.z += s.z; t.w += s.w;
    }
    cta_colsum(t, lq, colsum);
}

}  // namespace dst_nn
