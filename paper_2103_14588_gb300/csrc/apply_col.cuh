// 3+1 operator apply with blocks of 2 x 4 outputs (y, z) per thread column: large meshes
// whose nodes all have the standard interior stencils (periodic or Dirichlet axes) and
// whose potential depends on x only or vanishes.
//
// Same operator as apply_pipe.cuh: Appendix A's element matrices summed into [1,4,1] /
// [-1,0,1] tensor stencils per time plane, combined with the spin matrices, then the two
// time stencils through running accumulators.  Time planes of the tile with a one-node
// halo are staged by cp.async, the next one while this one is summed.
//
// What bounds it: FP32 the issue slots and shared-memory loads, FP64 the FP64 pipe (1/64 of
// the FP32 rate).  So each thread keeps as many sums to itself as its registers hold: it
// walks the six z slices of its column, forms the x sums of four rows once for two y
// outputs, and completes an output's z sums from the window of the last three slices.
// The stencils act on each spinor component alone and alpha_k couples components c with
// 3 - c (x, y) and c ^ 2 (z), so a column is shared by two lanes of two components (FP32) or
// four of one (FP64), 16 bytes of a node each, which exchange convection fields by
// shuffles.  In FP32 the real and imaginary part go through one packed instruction
// (f32x2): half the issue slots of the sums.
// 48^4 Klein mesh: FP32 100 us, 163 with columns of one output in y and z apart (two CTAs per SM
// without spills; three, with 100 bytes spilled, 136), FP64 2.94 ms, 4.79 so (33 FP64
// instructions per real output and plane, 46 so; 2.4 ms at the pipe's rate).
#pragma once

#include "apply_pipe.cuh"

namespace dst {

// Complex pairs: packed FP32 instructions, or two FP64 ones.
__device__ __forceinline__ unsigned long long pk(float2 a) { return *reinterpret_cast<unsigned long long *>(&a); }
__device__ __forceinline__ float2 up(unsigned long long a) { return *reinterpret_cast<float2 *>(&a); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return up(d);
}
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)), "l"(pk(c)));
    return up(d);
}
__device__ __forceinline__ float2 vmul(float2 a, float2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return up(d);
}
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return vfma(make_float2(-1.f, -1.f), b, a); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 vsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}

template <typename T>
struct ColShape {
    static constexpr int TX = 16, TY = 8, RY = 2, RZ = 4;
    static constexpr int LANES = sizeof(T) == 4 ? 2 : 4, COMPS = 4 / LANES;    // lanes per column, components per lane
    static constexpr int BX = TX + 2, BY = TY + 2, BZ = RZ + 2, BOX = BX * BY * BZ;
    static constexpr int NODE_BYTES = 8 * (int)sizeof(T), CHUNKS = NODE_BYTES / 16;
    static constexpr int NTHR = TX * (TY / RY) * LANES, CTAS = sizeof(T) == 4 ? 2 : 1;
    static constexpr int SLOT = BOX * NODE_BYTES, STAGES = 2;
    static constexpr int SMEM = STAGES * SLOT + BOX * (int)sizeof(int);
};

// Sums over x and y of one z slice, for the thread's two y outputs.
template <typename V, int COMPS>
struct ColFields {
    V M[2][COMPS], Cx[2][COMPS], Cy[2][COMPS];
};

// WV: x-only potential (see fields_std of apply_pipe.cuh); else none.
template <typename T, bool WV>
__global__ void __launch_bounds__(ColShape<T>::NTHR, ColShape<T>::CTAS)
apply_col_kernel(OpParams p, StdConst<T> sc, const typename C2<T>::type *__restrict__ x, typename C2<T>::type *__restrict__ y,
                 int tiles_x, int tiles_y, int64_t units) {
    using S = ColShape<T>;
    using V = typename C2<T>::type;
    using F = ColFields<V, S::COMPS>;
    constexpr int NC = S::COMPS, RY = S::RY, RZ = S::RZ;
    extern __shared__ __align__(16) char smc[];
    int *src_tab = reinterpret_cast<int *>(smc + S::STAGES * S::SLOT);
    const int h = threadIdx.x % S::LANES, col = threadIdx.x / S::LANES;
    const int tx = col % S::TX, ty = col / S::TX * RY;
    const int64_t nx = p.ax[0].n, ny = p.ax[1].n, nz = p.ax[2].n, N = p.nt;
    auto both = [](T a, T b) { V v; v.x = a; v.y = b; return v; };
    const V four = both(4, 4);
    // FP64: signs of the lane's component
    const T s1 = h & 1 ? -sc.ka[1] : sc.ka[1], s2 = h & 1 ? -sc.ka[2] : sc.ka[2];
    const int64_t plane_elems = nx * ny * nz * 4;
    const size_t plane_bytes = (size_t)plane_elems * sizeof(V);
    // the CTA's share of all layers of all tiles, in runs of one tile
    const int64_t end = units * (blockIdx.x + 1LL) / gridDim.x;
    for (int64_t at = units * blockIdx.x / gridDim.x, len; at < end; at += len) {
        const int tile = (int)(at / N);
        const int64_t t0 = 1 + at % N;
        len = min(N + 1 - t0, end - at);
        const int64_t t1 = t0 + len, pfirst = t0 - 1;
        const int64_t x0 = (int64_t)(tile % tiles_x) * S::TX, y0 = (int64_t)((tile / tiles_x) % tiles_y) * S::TY,
                      z0 = (int64_t)(tile / (tiles_x * tiles_y)) * RZ;
        const int64_t ix = x0 + tx, iy = y0 + ty;
        __syncthreads();                                   // the ring and the table of the run before are read
        // copy sources of the box (byte offset in a layer, -1 outside a wall)
        for (int b = threadIdx.x; b < S::BOX; b += S::NTHR) {
            const int bx = b % S::BX, by = (b / S::BX) % S::BY, bz = b / (S::BX * S::BY);
            const int gx = axis_nbr32(p.ax[0], (int)x0 - 1 + bx), gy = axis_nbr32(p.ax[1], (int)y0 - 1 + by),
                      gz = axis_nbr32(p.ax[2], (int)z0 - 1 + bz);
            src_tab[b] = (gx >= 0 && gy >= 0 && gz >= 0) ? ((gz * (int)ny + gy) * (int)nx + gx) * S::NODE_BYTES : -1;
        }
        // factors of the lane's components: beta is +1 for components 0, 1 and -1 for 2, 3
        const bool pos = NC * h < 2;
        T wa = pos ? -(T)p.m * sc.km : (T)p.m * sc.km, wb = 0;
        if (WV && ix < nx) {
            const int64_t g = ix + p.ax[0].u0, nel = p.ax[0].nel;
            const double *w = p.wx + (pos ? 0 : nel);
            const T wl = (T)w[g > 0 ? g - 1 : nel - 1], wr = (T)w[g < nel ? g : 0];
            wa = (T)-0.5 * sc.km * (wl + wr);
            wb = (T)-0.5 * sc.km * (wr - wl);
        }
        const V a2 = both(wa, wa), b2 = both(wb, wb);
        const int nplanes = (int)(t1 - t0 + 2);            // planes t0 - 1 .. t1
        const int i_lo = (int)max((int64_t)0, 1 - pfirst), i_hi = (int)min((int64_t)(nplanes - 1), N - pfirst);
        const int i_last = (int)(N - pfirst);
        const char *issue_src = reinterpret_cast<const char *>(x) + (pfirst - 1) * (int64_t)plane_bytes;
        __syncthreads();
        auto issue = [&](int i) {
            if (i >= i_lo && i <= i_hi) {
                char *slot = smc + (i & 1) * S::SLOT;
#pragma unroll 4
                for (int j = threadIdx.x; j < S::BOX * S::CHUNKS; j += S::NTHR) {
                    const int so = src_tab[j / S::CHUNKS];
                    cp_async16(slot + j * 16, issue_src + (so >= 0 ? so : 0) + j % S::CHUNKS * 16, so >= 0);
                }
            }
            cp_async_commit();
            issue_src += plane_bytes;
        };
        V accP[RZ][RY][NC], accC[RZ][RY][NC];
#pragma unroll
        for (int r = 0; r < RZ; ++r)
#pragma unroll
            for (int q = 0; q < RY; ++q)
#pragma unroll
                for (int l = 0; l < NC; ++l) { accP[r][q][l] = cz<V>(); accC[r][q][l] = cz<V>(); }
        char *ydst = reinterpret_cast<char *>(y + (t0 - 1) * plane_elems + ((z0 * ny + iy) * nx + ix) * 4 + NC * h);
        const size_t ystride = (size_t)nx * 4 * sizeof(V), zstride = ystride * ny;
        const int cbase = ty * S::BX + tx;                 // box node (x - 1, y - 1) of the first output
        issue(0);
        for (int i = 0; i < nplanes; ++i) {
            cp_async_wait<0>();
            __syncthreads();
            issue(i + 1);
            const bool have = i >= i_lo && i <= i_hi, last = i >= i_last;
            const char *slot = smc + (i & 1) * S::SLOT + 16 * h;
            // the sums of a slice's four rows and two outputs
            auto slice = [&](int bz, F &f) {
                V rM[RY + 2][NC], rC[RY + 2][NC];
#pragma unroll
                for (int q = 0; q < RY + 2; ++q) {
                    V n[3][NC];
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        const char *at = slot + ((bz * S::BY + q) * S::BX + cbase + dx) * S::NODE_BYTES;
                        if constexpr (NC == 2) {
                            const float4 v = *reinterpret_cast<const float4 *>(at);
                            n[dx][0] = both(v.x, v.y);
                            n[dx][1] = both(v.z, v.w);
                        } else {
                            n[dx][0] = *reinterpret_cast<const V *>(at);
                        }
                    }
#pragma unroll
                    for (int l = 0; l < NC; ++l) {
                        rM[q][l] = vfma(four, n[1][l], vadd(n[0][l], n[2][l]));
                        rC[q][l] = vsub(n[2][l], n[0][l]);
                    }
                }
#pragma unroll
                for (int q = 0; q < RY; ++q)
#pragma unroll
                    for (int l = 0; l < NC; ++l) {
                        f.M[q][l] = vfma(four, rM[q + 1][l], vadd(rM[q][l], rM[q + 2][l]));
                        f.Cx[q][l] = vfma(four, rC[q + 1][l], vadd(rC[q][l], rC[q + 2][l]));
                        f.Cy[q][l] = vsub(rM[q + 2][l], rM[q][l]);
                    }
            };
            F w0, w1, w2;
#pragma unroll
            for (int bz = 0; bz < RZ + 2; ++bz) {
                F &C = bz % 3 == 0 ? w0 : (bz % 3 == 1 ? w1 : w2);
                if (have) slice(bz, C);
                if (bz < 2) continue;
                const F &A = (bz - 2) % 3 == 0 ? w0 : ((bz - 2) % 3 == 1 ? w1 : w2), &B = (bz - 1) % 3 == 0 ? w0 : ((bz - 1) % 3 == 1 ? w1 : w2);
                const int r = bz - 2;
#pragma unroll
                for (int q = 0; q < RY; ++q) {
                    V GM[NC], QM[NC], QX[NC], QY[NC], QZ[NC];
                    if (have) {
#pragma unroll
                        for (int l = 0; l < NC; ++l) {
                            QM[l] = vadd(vfma(four, B.M[q][l], A.M[q][l]), C.M[q][l]);
                            QX[l] = vadd(vfma(four, B.Cx[q][l], A.Cx[q][l]), C.Cx[q][l]);
                            QY[l] = vadd(vfma(four, B.Cy[q][l], A.Cy[q][l]), C.Cy[q][l]);
                            QZ[l] = vsub(C.M[q][l], A.M[q][l]);
                            GM[l] = vmul(a2, QM[l]);
                            if (WV) GM[l] = vfma(b2, QX[l], GM[l]);
                        }
                        // i alpha
                        if constexpr (NC == 2) {
                            // both partner components sit in lane ^ 1: this lane forms what its components add to
                            // them (of component l there: 1 - l here along x and y, l along z) and sends the sums
                            V E[2];
#pragma unroll
                            for (int l = 0; l < 2; ++l) {
                                const float s1 = l ? -sc.ka[1] : sc.ka[1], s2 = l ? -sc.ka[2] : sc.ka[2];
                                E[l].x = fmaf(-s2, QZ[l].y, fmaf(-sc.ka[0], QX[1 - l].y, s1 * QY[1 - l].x));
                                E[l].y = fmaf(s2, QZ[l].x, fmaf(sc.ka[0], QX[1 - l].x, s1 * QY[1 - l].y));
                            }
#pragma unroll
                            for (int l = 0; l < 2; ++l)
                                GM[l] = vadd(GM[l], both(__shfl_xor_sync(0xffffffffu, E[l].x, 1), __shfl_xor_sync(0xffffffffu, E[l].y, 1)));
                        } else {
                            // shuffles are cheaper than FP64 instructions: the fields themselves
                            const V X = both(__shfl_xor_sync(0xffffffffu, QX[0].y, 3), __shfl_xor_sync(0xffffffffu, QX[0].x, 3));
                            const V Y = both(__shfl_xor_sync(0xffffffffu, QY[0].x, 3), __shfl_xor_sync(0xffffffffu, QY[0].y, 3));
                            const V Z = both(__shfl_xor_sync(0xffffffffu, QZ[0].y, 2), __shfl_xor_sync(0xffffffffu, QZ[0].x, 2));
                            GM[0] = vfma(both(-s2, s2), Z, vfma(both(s1, s1), Y, vfma(both(-sc.ka[0], sc.ka[0]), X, GM[0])));
                        }
                    } else {
#pragma unroll
                        for (int l = 0; l < NC; ++l) { GM[l] = cz<V>(); QM[l] = cz<V>(); }
                    }
                    // with G_C' = i kc QM: y(pl-1) += G_C' + G_M'; y(pl) += (pl < N ? 4 G_M' : G_C' + 2 G_M');
                    // y(pl+1) = G_M' - G_C'
                    char *at = ydst + r * zstride + q * ystride;
                    const bool store = i >= 2 && ix < nx && iy + q < ny && z0 + r < nz;
                    V out[NC];
#pragma unroll
                    for (int l = 0; l < NC; ++l) {
                        const V t = vadd(accP[r][q][l], GM[l]);
                        out[l] = both(fma(-sc.kc, QM[l].y, t.x), fma(sc.kc, QM[l].x, t.y));
                        accP[r][q][l] = vfma(four, GM[l], accC[r][q][l]);
                        if (last) {
                            const V u = vfma(both(2, 2), GM[l], accC[r][q][l]);
                            accP[r][q][l] = both(fma(-sc.kc, QM[l].y, u.x), fma(sc.kc, QM[l].x, u.y));
                        }
                        accC[r][q][l] = both(fma(sc.kc, QM[l].y, GM[l].x), fma(-sc.kc, QM[l].x, GM[l].y));
                    }
                    if (store) {
                        if constexpr (NC == 2)
                            *reinterpret_cast<float4 *>(at) = make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
                        else
                            *reinterpret_cast<V *>(at) = out[0];
                    }
                }
            }
            if (i >= 2) ydst += plane_bytes;
        }
        cp_async_wait<0>();
    }
}

// CTAs of the launch: as many as are resident at once, each with an equal share of the
// (tile, layer) units in order, so that none waits for a last wave.  A run of layers of one
// tile sums two planes beyond its own, so no share is shorter than four.  Variant 1 of the
// tile autotuner launches twice as many.
template <typename T>
inline int64_t col_ctas(int64_t units, int variant) {
    const int64_t slots = 152LL * ColShape<T>::CTAS * (variant == 1 ? 2 : 1);
    return std::max<int64_t>(1, std::min(slots, units / 4));
}

template <typename T>
int launch_apply_col(const OpParams &p, const typename C2<T>::type *x, typename C2<T>::type *y, cudaStream_t s) {
    using S = ColShape<T>;
    const int64_t tx = (p.ax[0].n + S::TX - 1) / S::TX, ty = (p.ax[1].n + S::TY - 1) / S::TY,
                  tz = (p.ax[2].n + S::RZ - 1) / S::RZ, tiles = tx * ty * tz;
    // byte offsets within one time layer are kept in 32 bits
    if (p.ax[0].n * p.ax[1].n * p.ax[2].n * S::NODE_BYTES >= (1LL << 31)) return launch_apply_node<3, 4, T>(p, x, y, s);
    const int64_t units = tiles * p.nt;
    const int64_t ctas = col_ctas<T>(units, p.tile_variant[sizeof(T) == 4 ? DST_FP32 : DST_FP64]);
    static bool configured[2][DST_MAX_DEVICES_APPLY] = {};
    int dev = 0;
    DST_CUDA_TRY(cudaGetDevice(&dev));
    const int nov = p.vmode == 2 ? 1 : 0;
    auto kern = nov ? apply_col_kernel<T, false> : apply_col_kernel<T, true>;
    if (dev < 0 || dev >= DST_MAX_DEVICES_APPLY || !configured[nov][dev]) {
        DST_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM));
        if (dev >= 0 && dev < DST_MAX_DEVICES_APPLY) configured[nov][dev] = true;
    }
    kern<<<(unsigned)ctas, S::NTHR, S::SMEM, s>>>(p, std_const<3, T>(p), x, y, (int)tx, (int)ty, units);
    DST_CUDA_TRY(cudaGetLastError());
    return DST_OK;
}

}  // namespace dst
