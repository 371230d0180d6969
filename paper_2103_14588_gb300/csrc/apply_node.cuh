// Operator apply with a lane per number of a plane: every mesh
// (open axes, general potentials, planes of any size), and the choice where the tiled
// kernels are held back by their tiles.
//
// Same operator as apply_pipe.cuh: per time plane the [1,4,1] / [-1,0,1] tensor stencils of
// Appendix A's element matrices, the spin combination, the two time stencils through
// running accumulators.  The stencils are real, so in FP64 a lane takes the real or the imaginary
// part of one component (LaneOf); a node's lanes are neighbours and exchange their convection
// fields by shuffles, and every load is a plain run of numbers.  Nodes are taken in flat
// order, so a ragged mesh leaves no thread of a tile idle, and the chunk of time layers
// per thread is chosen at launch: it is what a small mesh fills the GPU with.
//
// What bounds it in FP64 is the FP64 pipe (two lanes per clock and SM, 1/64 of the FP32
// rate), so the sums are written for the fewest FP64 instructions and the neighbours come
// straight through L1; nothing is staged.  At the end node of an open axis an element is
// missing: its neighbour enters the mass sums as zero and the convection difference as
// the node itself, which selects, not multiplications, take care of.
// A general potential needs the mass sums of the 2^d elements around a node apart (four
// more operations per x row pair), the x-only one (w_l + w_r)/2 M + (w_r - w_l)/2 C.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "apply_impl.cuh"

namespace dst {

// One axis at one node: offsets of the neighbours (of the node itself where there is
// none), whether they hold a value, and which elements exist.
template <typename T>
struct AxisEnds {
    int64_t lo, hi;        // offsets in nodes from the node
    bool vl, vr;           // neighbour is an unknown (else its value is 0)
    bool el, er;           // element exists
    T wc;                  // centre weight of the mass sum: 2 per element
};
template <typename T, bool OPEN>
__device__ __forceinline__ AxisEnds<T> axis_ends(const AxisDesc &a, int64_t i, int64_t stride) {
    AxisEnds<T> e;
    const bool wrap = a.bc == DST_BC_PERIODIC, first = i == 0, last = i == a.n - 1;
    e.vl = wrap || !first;
    e.vr = wrap || !last;
    e.lo = first ? (wrap ? (a.n - 1) * stride : 0) : -stride;
    e.hi = last ? (wrap ? -(a.n - 1) * stride : 0) : stride;
    e.el = !OPEN || a.bc != DST_BC_OPEN || i > 0;
    e.er = !OPEN || a.bc != DST_BC_OPEN || i < a.n - 1;
    e.wc = (T)(2 * ((e.el ? 1 : 0) + (e.er ? 1 : 0)));
    return e;
}

// What a lane holds: one real number (FP64) or one complex number (FP32, where a lane's
// work is a few instructions and the wider load pays: the 96 x 96 x 96 mesh with an open
// axis takes 14.5 us so and 21.2 us with real lanes).
template <typename T> struct LaneOf;
template <> struct LaneOf<double> { using type = double; static constexpr int PER = 2; };   // lanes per complex number
template <> struct LaneOf<float> { using type = float2; static constexpr int PER = 1; };

__device__ __forceinline__ double ladd(double a, double b) { return a + b; }
__device__ __forceinline__ double lsub(double a, double b) { return a - b; }
__device__ __forceinline__ double lmul(double k, double a) { return k * a; }
__device__ __forceinline__ double lfma(double k, double a, double b) { return fma(k, a, b); }
__device__ __forceinline__ double lpick(bool b, double v, double w) { return b ? v : w; }
__device__ __forceinline__ float2 ladd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 lsub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 lmul(float k, float2 a) { return make_float2(k * a.x, k * a.y); }
__device__ __forceinline__ float2 lfma(float k, float2 a, float2 b) { return make_float2(fmaf(k, a.x, b.x), fmaf(k, a.y, b.y)); }
__device__ __forceinline__ float2 lpick(bool b, float2 v, float2 w) { return make_float2(b ? v.x : w.x, b ? v.y : w.y); }
// g + k f and g + i k f, f the value of component c ^ m; sg: -1 on lanes of a real part, 1 of an imaginary one
__device__ __forceinline__ double add_of(double g, double k, double v, int m, double) {
    return fma(k, __shfl_xor_sync(0xffffffffu, v, 2 * m), g);
}
__device__ __forceinline__ double add_i_of(double g, double k, double v, int m, double sg) {
    return fma(sg * k, __shfl_xor_sync(0xffffffffu, v, 2 * m | 1), g);
}
__device__ __forceinline__ float2 lane_of(float2 v, int m) {
    return m ? make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m)) : v;
}
__device__ __forceinline__ float2 add_of(float2 g, float k, float2 v, int m, float) { return lfma(k, lane_of(v, m), g); }
__device__ __forceinline__ float2 add_i_of(float2 g, float k, float2 v, int m, float) {
    const float2 f = lane_of(v, m);
    return make_float2(fmaf(-k, f.y, g.x), fmaf(k, f.x, g.y));
}

// VM: 0 x-only potential, 1 general, 2 none (OpParams::vmode).  OPEN: some axis is open (else
// every element exists and the selects fall away).
template <int D, int NC, typename T, int VM, bool OPEN>
__global__ void __launch_bounds__(128)
apply_node_kernel(OpParams p, StdConst<T> sc, int tt, const typename LaneOf<T>::type *__restrict__ x,
                  typename LaneOf<T>::type *__restrict__ y) {
    using V = typename LaneOf<T>::type;
    constexpr int NY = D >= 2 ? 3 : 1, NZ = D >= 3 ? 3 : 1, R = LaneOf<T>::PER * NC;   // R: lanes per node
    const V zero = {};
    const int64_t nx = p.ax[0].n, ny = p.ax[1].n, plane = nx * ny * p.ax[2].n;
    const int64_t id = blockIdx.x * 128LL + threadIdx.x;
    const bool valid = id < plane * R;                     // lanes past the mesh work on its first node
    const int lane = threadIdx.x % R, c = lane / LaneOf<T>::PER;
    const int64_t s = valid ? id / R : 0;
    int64_t ix = s, iy = 0, iz = 0;
    if (D >= 2) {
        if (plane <= 0x7fffffff) {
            const unsigned row = (unsigned)s / (unsigned)nx;
            ix = (unsigned)s - row * (unsigned)nx;
            iz = D >= 3 ? row / (unsigned)ny : 0u;
            iy = row - (unsigned)iz * (unsigned)ny;
        } else {
            const int64_t row = s / nx;
            ix = s - row * nx;
            iz = D >= 3 ? row / ny : 0;
            iy = row - iz * ny;
        }
    }
    const AxisEnds<T> ex = axis_ends<T, OPEN>(p.ax[0], ix, R);
    AxisEnds<T> ey = {}, ez = {};
    if (D >= 2) ey = axis_ends<T, OPEN>(p.ax[1], iy, nx * R);
    if (D >= 3) ez = axis_ends<T, OPEN>(p.ax[2], iz, nx * ny * R);
    const int64_t oy[3] = {ey.lo, 0, ey.hi}, oz[3] = {ez.lo, 0, ez.hi};
    const bool vy[3] = {ey.vl, true, ey.vr}, vz[3] = {ez.vl, true, ez.vr};
    // beta of the component; factors of the mass and potential sums, times -(h_t/6) prod h/6
    const bool up = c < NC / 2;
    T wm = 0, wb = 0, vc[8];
    if (VM == 2) {
        wm = up ? (T)-p.m * sc.km : (T)p.m * sc.km;
    } else if (VM == 0) {
        const int64_t g = ix + p.ax[0].u0, nel = p.ax[0].nel;
        const double *w = p.wx + (up ? 0 : nel);
        const T wl = ex.el ? (T)w[g > 0 ? g - 1 : nel - 1] : (T)0, wr = ex.er ? (T)w[g < nel ? g : 0] : (T)0;
        const T h = ex.el && ex.er ? (T)-0.5 : (T)-1;
        wm = h * sc.km * (wl + wr);
        wb = ex.el && ex.er ? (T)-0.5 * sc.km * (wr - wl) : (T)0;
    } else {
        const T m = up ? (T)p.m : (T)-p.m;
        auto elem = [&](const AxisDesc &a, int64_t i, int side) {
            const int64_t g = i + a.u0 - 1 + side;
            return a.bc == DST_BC_PERIODIC && g < 0 ? g + a.nel : g;
        };
#pragma unroll
        for (int k = 0; k < 1 << D; ++k) {
            const int sx = k & 1, sy = (k >> 1) & 1, sz = (k >> 2) & 1;
            const bool ok = (sx ? ex.er : ex.el) && (D < 2 || (sy ? ey.er : ey.el)) && (D < 3 || (sz ? ez.er : ez.el));
            const int64_t e0 = elem(p.ax[0], ix, sx), e1 = D >= 2 ? elem(p.ax[1], iy, sy) : 0,
                          e2 = D >= 3 ? elem(p.ax[2], iz, sz) : 0;
            vc[k] = ok ? -sc.km * (m + (T)p.Vel[(e2 * p.ax[1].nel + e1) * p.ax[0].nel + e0]) : (T)0;
        }
    }
    const T sg = lane & 1 ? (T)1 : (T)-1;
    const T k1 = c & 1 ? -sc.ka[1] : sc.ka[1], k2 = c & 1 ? -sc.ka[2] : sc.ka[2];
    const int64_t N = p.nt, t0 = 1 + blockIdx.y * (int64_t)tt, t1 = min(t0 + (int64_t)tt, N + 1);
    const int64_t step = plane * R;
    // planes t0 - 1 .. t1 of x, without the layers 0 and N + 1, which hold nothing, but where
    // bounds of their own cost the loop registers (48^4 elements with an open axis, FP32:
    // 390 us as zeros, 422 so)
    constexpr bool TRIM = !(D == 3 && sizeof(T) == 4 && OPEN && VM != 1);
    const int64_t tb = TRIM ? max(t0 - 1, (int64_t)1) : t0 - 1, te = TRIM ? min(t1, N) : t1;
    const V *src = x + (tb - 1) * step + s * R + lane;
    V *dst = y + (t0 - 1) * step + s * R + lane;
    V accP = zero, accC = zero;
    struct Rows { V v[NY][3]; };
    auto load = [&](const V *at, bool have, int dz, Rows &r) {
#pragma unroll
        for (int dy = 0; dy < NY; ++dy) {
            const bool ok = have && (D < 2 || vy[dy]) && (D < 3 || vz[dz]);
            const V *q = at + (D >= 2 ? oy[dy] : 0) + (D >= 3 ? oz[dz] : 0);
            r.v[dy][0] = ok && ex.vl ? __ldg(q + ex.lo) : zero;
            r.v[dy][1] = ok ? __ldg(q) : zero;
            r.v[dy][2] = ok && ex.vr ? __ldg(q + ex.hi) : zero;
        }
    };
    auto mass = [](V l, T wc, V m, V r) { return lfma(wc, m, ladd(l, r)); };
    auto diff = [](bool lo, V l, V m, V r, bool hi) { return lsub(lpick(hi, r, m), lpick(lo, l, m)); };
    auto half = [&](bool ok, V m, V o) { return lpick(ok, lfma((T)2, m, o), zero); };
    // with one or nine neighbours the next plane's loads run ahead of this plane's sums
    Rows cur;
    if (D < 3) load(src, true, 0, cur);
    for (int64_t t = tb; t <= te; ++t, src += step) {
        Rows nxt;
        if (D < 3) load(src + step, t < te, 0, nxt);
        // sums over x and y of each z slice, then over z: mass, convection along x, y, z,
        // and for a general potential the mass sums of the elements on the eight sides
        V M, Cx, Cy = zero, Cz = zero, W = zero, Mz[3], Xz[3], Yz[3], Q[3][4];
#pragma unroll
        for (int dz = 0; dz < NZ; ++dz) {
            // (with TRIM the condition always holds; it keeps the loads predicated: 5 x 40 x 40 x 60
            // elements with an open axis, FP64, 541 us, 654 without)
            if (D == 3) load(src, t >= 1 && t <= N, dz, cur);
            V rM[NY], rC[NY], L[NY], H[NY];
#pragma unroll
            for (int dy = 0; dy < NY; ++dy) {
                const V a = cur.v[dy][0], b = cur.v[dy][1], d = cur.v[dy][2];
                rC[dy] = diff(ex.el, a, b, d, ex.er);
                if (VM == 1) {
                    L[dy] = half(ex.el, b, a);
                    H[dy] = half(ex.er, b, d);
                    rM[dy] = ladd(L[dy], H[dy]);
                } else {
                    rM[dy] = mass(a, ex.wc, b, d);         // a missing neighbour was loaded as zero
                }
            }
            if (D == 1) {
                Mz[dz] = rM[0]; Xz[dz] = rC[0];
                if (VM == 1) { Q[dz][0] = L[0]; Q[dz][1] = H[0]; }
            } else {
                Mz[dz] = mass(rM[0], ey.wc, rM[1], rM[2]);
                Xz[dz] = mass(rC[0], ey.wc, rC[1], rC[2]);
                Yz[dz] = diff(ey.el, rM[0], rM[1], rM[2], ey.er);
                if (VM == 1) {
                    Q[dz][0] = half(ey.el, L[1], L[0]); Q[dz][1] = half(ey.el, H[1], H[0]);
                    Q[dz][2] = half(ey.er, L[1], L[2]); Q[dz][3] = half(ey.er, H[1], H[2]);
                }
            }
        }
        if (D < 3) {
            M = Mz[0]; Cx = Xz[0];
            if (D == 2) Cy = Yz[0];
            if (VM == 1) {
#pragma unroll
                for (int k = 0; k < 1 << D; ++k) W = lfma(vc[k], Q[0][k], W);
            }
        } else {
            M = mass(Mz[0], ez.wc, Mz[1], Mz[2]);
            Cx = mass(Xz[0], ez.wc, Xz[1], Xz[2]);
            Cy = mass(Yz[0], ez.wc, Yz[1], Yz[2]);
            Cz = diff(ez.el, Mz[0], Mz[1], Mz[2], ez.er);
            if (VM == 1) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    W = lfma(vc[k], half(ez.el, Q[1][k], Q[0][k]), W);
                    W = lfma(vc[4 + k], half(ez.er, Q[1][k], Q[2][k]), W);
                }
            }
        }
        const V GC = add_i_of(zero, sc.kc, M, 0, sg);
        V GM = VM == 1 ? W : VM == 0 ? lfma(wb, Cx, lmul(wm, M)) : lmul(wm, M);
        // i alpha: x takes component 1 - c (3 - c), y its (-i, i) multiple, z (3+1) the (1, -1) multiple of c ^ 2
        constexpr int PX = NC == 2 ? 1 : 3;
        GM = add_i_of(GM, sc.ka[0], Cx, PX, sg);
        if (D >= 2) GM = add_of(GM, k1, Cy, PX, sg);
        if (D >= 3) GM = add_i_of(GM, k2, Cz, 2, sg);
        // y(t-1) += GC + GM; y(t) += (t < N ? 4 GM : GC + 2 GM); y(t+1) = GM - GC
        accP = ladd(accP, ladd(GC, GM));
        accC = t < N ? lfma((T)4, GM, accC) : ladd(accC, lfma((T)2, GM, GC));
        if (t > t0) {
            if (valid) *dst = accP;
            dst += step;
        }
        accP = accC;
        accC = lsub(GM, GC);
        if (D < 3) cur = nxt;
    }
    if (valid && te < t1) *dst = accP;                     // the last layer
}

// Layers per thread.  Each chunk forms the sums of two planes that its neighbours form
// too, so long chunks save work, but a mesh of few nodes needs its layers spread.
// FP64: a warp's instruction holds one of the 608 FP64 units for 64 clocks, so the time is
// the planes of a chunk times the warps that share a unit (a CTA's four warps, working or
// not, sit on four units); the chunk with the least (1+1, 520 x 520: 31 us with 20 layers, 53 with
// the 58 that a count of the working warps alone would take).
// FP32: latency; the longest chunk that leaves 12 warps per SM (16 x 16 x 16 x 16 elements
// 3+1: 17.2 / 11.4 / 10.1 / 11.5 us with 3 / 6 / 12 / 24).
template <typename T>
inline int node_chunk(int64_t plane_threads, int64_t nt) {
    if (sizeof(T) == 4) {
        const int64_t warps = (plane_threads + 31) / 32;
        int64_t chunks = (152 * 12 + warps - 1) / warps;
        chunks = std::min<int64_t>(std::max<int64_t>(chunks, (nt + 31) / 32), nt);
        return (int)((nt + chunks - 1) / chunks);
    }
    const int64_t warps = (plane_threads + 127) / 128 * 4;
    // a unit's share, rounded up to whole warps while they are few (the sum then follows the
    // measured times of 31 meshes to within 7%)
    auto time = [&](int64_t tt) {
        const double share = (double)(warps * ((nt + tt - 1) / tt)) / 608.0;
        return (double)std::min(tt + 2, nt) * (share > 4.0 ? share + 0.5 : std::ceil(share));
    };
    int64_t best = nt;
    for (int64_t tt = 1; tt < std::min<int64_t>(nt, 64); ++tt)
        if (time(tt) < time(best)) best = tt;
    return (int)std::min<int64_t>(best, 1 << 20);
}

// Where the tiled kernels (apply_pipe.cuh and what builds on it) take over: every node with
// the standard stencils, an x-only or no potential, and enough unknowns for their tiles to
// fill the GPU.  Measured on both sides of 2^19 unknowns: 1+1 FP32 512^2 4.5 us here, 6.0
// tiled, 1024^2 11.6 and 7.9; 2+1 FP32 48^3 3.7 and 6.2, 64^3 7.4 and 4.9, 96^3 16.2 and
// 9.2, FP64 64^3 72 and 66; 3+1 FP32 16^4 8.7 and 25.4, 24^4 27 and 20, FP64 24^4 354 and 331.  Meshes with an open
// axis stay here at every size (2+1 96^3 FP32 14.5 us, 37.7 tiled).
template <int D>
inline bool tiles_pay(const OpParams &p) {
    if (p.vmode == 1) return false;
    for (int k = 0; k < D; ++k)
        if (p.ax[k].bc == DST_BC_OPEN) return false;
    return p.ax[0].n * p.ax[1].n * p.ax[2].n * p.nt * (D == 3 ? 4 : 2) >= 1 << 19;
}

template <int D, int NC, typename T>
int launch_apply_node(const OpParams &p, const typename C2<T>::type *xv, typename C2<T>::type *yv, cudaStream_t s) {
    using V = typename LaneOf<T>::type;
    const V *x = reinterpret_cast<const V *>(xv);
    V *y = reinterpret_cast<V *>(yv);
    const int64_t threads = p.ax[0].n * p.ax[1].n * p.ax[2].n * NC * LaneOf<T>::PER, blocks = (threads + 127) / 128;
    int tt = node_chunk<T>(threads, p.nt);
    if ((p.nt + tt - 1) / tt > 65535) tt = (int)((p.nt + 65534) / 65535);
    const int64_t chunks = (p.nt + tt - 1) / tt;
    if (blocks <= 0 || blocks > 0x7fffffffLL || chunks > 65535) return DST_ERR_ARG;
    const dim3 grid((unsigned)blocks, (unsigned)chunks);
    const StdConst<T> sc = std_const<D, T>(p);
    bool open = false;
    for (int k = 0; k < D; ++k) open = open || p.ax[k].bc == DST_BC_OPEN;
    auto go = [&](auto vm) {
        constexpr int VM = decltype(vm)::value;
        if (open) apply_node_kernel<D, NC, T, VM, true><<<grid, 128, 0, s>>>(p, sc, tt, x, y);
        else apply_node_kernel<D, NC, T, VM, false><<<grid, 128, 0, s>>>(p, sc, tt, x, y);
    };
    if (p.vmode == 0) go(std::integral_constant<int, 0>());
    else if (p.vmode == 1) go(std::integral_constant<int, 1>());
    else go(std::integral_constant<int, 2>());
    DST_CUDA_TRY(cudaGetLastError());
    return DST_OK;
}

}  // namespace dst
