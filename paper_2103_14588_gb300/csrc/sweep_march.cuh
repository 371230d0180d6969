// The Crank-Nicolson march of the sweep along a Dirichlet x axis (sweep.cu, banded
// mode): x_t = Bd^-1 (s_t - Bl x_{t-1}) for every frequency of the periodic axes.
//
// Three identities shape the kernels.
// 1. Bd + Bl = h_t K, so the increment u_t = x_t - x_{t-1} solves
//    Bd u_t = s_t - h_t K x_{t-1}.  The rounding of the solve is then relative to the
//    increment, which is small for the modes that the time step resolves.
// 2. At one (y, z) frequency K contains alpha_y b_y + alpha_z b_z with the same x
//    mass.  The rotation exp(-i phi / 2 Sigma_x), tan phi = b_z / b_y, commutes with
//    alpha_x and beta and turns it into alpha_y P, P = |b|, which couples the spinor
//    components only within the pairs (0, 3) (as sigma_x, P sigma_y, sigma_z) and
//    (1, 2) (as sigma_x, -P sigma_y, sigma_z).  So a 3+1 frequency is two systems of
//    2 x 2 blocks, of the 2+1 kind, at a quarter of the block work each; and since
//    only |sin| enters P, the factors are shared by the frequencies +-k.
// 3. S^-1 also runs forward: s_0 = 2 sum_t (-1)^t v_t, s_{t+1} = 2 v_t - s_t.  With
//    s_0 from one reading pass (altsum_kernel) the time scan costs no pass of its own.
//
// The layer solve.  The systems are few (2 x 2304 for the 48^3 x 48 Klein mesh) and the
// time steps are a serial chain, so block Thomas elimination (a chain of 2 n_x small
// products per layer) leaves the GPU waiting (4.5 ms there, 0.25 so).  Here G lanes share a
// system, two x nodes each: one cyclic-reduction step removes the odd nodes, parallel
// cyclic reduction over the even ones needs log2(G) exchanges, and the odd nodes follow.
// Twice the arithmetic of the elimination, a seventh of the chain.  Bd = i M + (h_t/2) K
// with M positive definite and K Hermitian, so every Schur complement met on the way
// keeps a positive definite part (no pivoting).  The factors (2 x 2 blocks per lane and
// step) stay in registers for all layers when G <= 32.
// Layers stream through a shared-memory ring (cp.async), rows of neighbouring
// frequencies, so that global memory sees whole sectors although a warp walks along x.
#pragma once

#include "sweep.h"

namespace dst_march {

constexpr int STAGES = 3;                 // input layers in shared memory
constexpr int REG_STEPS = 5;              // reduction steps whose factors stay in registers (G <= 32)

// A pair of floats hi + lo (48 bits): the arithmetic of the factors.  The FP64 unit
// issues one warp instruction in 64 clocks, a product and a sum of pairs take 12 in FP32.
// Products are __fmul_rn so that they are not contracted into the sums that follow.
struct df { float h, l; };
__device__ __forceinline__ df to_df(double v) { const float h = (float)v; return df{h, (float)(v - (double)h)}; }
__device__ __forceinline__ df operator*(df a, df b) {
    const float p = __fmul_rn(a.h, b.h);
    return df{p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
}
__device__ __forceinline__ df operator+(df a, df b) {
    const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
    return df{s, (a.l + b.l) + (__fsub_rn(a.h, __fsub_rn(s, t)) + __fsub_rn(b.h, t))};
}
__device__ __forceinline__ df operator-(df a) { return df{-a.h, -a.l}; }
__device__ __forceinline__ df operator-(df a, df b) { return a + -b; }
__device__ __forceinline__ df scaled(df a, float power_of_2) { return df{a.h * power_of_2, a.l * power_of_2}; }
__device__ __forceinline__ df norm(df a) {                 // hi = the sum rounded
    const float s = __fadd_rn(a.h, a.l);
    return df{s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
}

struct z2 { df x, y; };
__device__ __forceinline__ z2 operator+(z2 a, z2 b) { return z2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ z2 operator-(z2 a, z2 b) { return z2{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ z2 operator-(z2 a) { return z2{-a.x, -a.y}; }
__device__ __forceinline__ z2 operator*(z2 a, z2 b) { return z2{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ z2 norm(z2 a) { return z2{norm(a.x), norm(a.y)}; }

struct M22 { z2 a, b, c, d; };            // rows (a b), (c d)
struct Row { z2 a, b; };                  // one row of a block
__device__ __forceinline__ Row norm(const Row &p) { return Row{norm(p.a), norm(p.b)}; }
__device__ __forceinline__ Row mul(const Row &p, const M22 &q) {
    return norm(Row{p.a * q.a + p.b * q.c, p.a * q.b + p.b * q.d});
}
__device__ __forceinline__ Row sub(const Row &p, const Row &q) { return norm(Row{p.a - q.a, p.b - q.b}); }
__device__ __forceinline__ Row neg(const Row &p) { return Row{-p.a, -p.b}; }
__device__ __forceinline__ Row row(const M22 &m, int h) { return h ? Row{m.c, m.d} : Row{m.a, m.b}; }
// Row h of the inverse of a block of which this lane has row h, the lane beside it the other
__device__ __forceinline__ Row inv_row(const Row &p, int h) {
    auto other = [](df v) { return df{__shfl_xor_sync(0xffffffffu, v.h, 1), __shfl_xor_sync(0xffffffffu, v.l, 1)}; };
    const Row o{z2{other(p.a.x), other(p.a.y)}, z2{other(p.b.x), other(p.b.y)}};
    // a d - b c, of either row the same
    z2 det = norm(h ? o.a * p.b - o.b * p.a : p.a * o.b - p.b * o.a);
    // the determinant scaled to [1, 2) by a power of two: its square stays in range
    const float big = fmaxf(fabsf(det.x.h), fabsf(det.y.h));
    const float sc = __int_as_float((254 << 23) - (__float_as_int(big) & 0x7f800000));
    det = z2{scaled(det.x, sc), scaled(det.y, sc)};
    const df n = norm(det.x * det.x + det.y * det.y);
    const float r0 = 1.f / n.h;
    const df r = norm(df{r0, r0 * fmaf(-n.l, r0, fmaf(-n.h, r0, 1.f))});      // a Newton step for 1 / n
    const z2 w{scaled(norm(det.x * r), sc), scaled(norm(-(det.y * r)), sc)}, m = -w;
    // (d -b; -c a) w
    return h ? norm(Row{p.a * m, o.a * w}) : norm(Row{o.b * w, p.b * m});
}

// Symbols of one frequency: prod of the y, z masses and the two transverse terms.
__device__ __forceinline__ void symbols(const SweepGeom &g, int i1, int i2, double &myz, double &by, double &bz) {
    // (sine and cosine of an angle come together: the FP64 unit is what these lines wait for)
    double s1 = 0.0, c1 = 1.0, s2 = 0.0, c2 = 1.0;
    if (g.ax1 >= 0) sincospi(2.0 * i1 / g.n1, &s1, &c1);
    if (g.ax2 >= 0) sincospi(2.0 * i2 / g.n2, &s2, &c2);
    const double sy = g.ax1 == 1 ? s1 : (g.ax2 == 1 ? s2 : 0.0), cy = g.ax1 == 1 ? c1 : (g.ax2 == 1 ? c2 : 1.0);
    const double sz = g.ax1 == 2 ? s1 : (g.ax2 == 2 ? s2 : 0.0), cz = g.ax1 == 2 ? c1 : (g.ax2 == 2 ? c2 : 1.0);
    const double my = g.d >= 2 ? g.h[1] * (2.0 + cy) * (1.0 / 3.0) : 1.0;
    const double mz = g.d >= 3 ? g.h[2] * (2.0 + cz) * (1.0 / 3.0) : 1.0;
    myz = my * mz;
    by = g.d >= 2 ? sy * mz : 0.0;
    bz = g.d >= 3 ? sz * my : 0.0;
}

// Distinct frequencies up to sign: classes (k1, k2), k = 0 .. n/2; each has a system for
// +P and one for -P (index 2 class + (P < 0)).
__host__ __device__ inline int class_count(int n1, int n2) { return (n1 / 2 + 1) * (n2 / 2 + 1); }

// A block of Bd at offset o from its x node, o in {-1, 0, 1}:
//   i M myz + (h_t/2) [ i C myz sigma_x - M P sigma_y - diag(W+, W-) myz ],
// from im = h/6 myz, c = h_t/4 myz, s = h_t/2 h/6 P, w = h_t/2 im and v, the potential of
// the element at that side (o = 0: 2 (left + right)).
struct BdSymbols { df im, c, s, w, m; };
__device__ __forceinline__ M22 bd_block(const BdSymbols &q, int o, df v) {
    const float k = o == 0 ? 4.f : 1.f;
    const df im = scaled(q.im, k), s = scaled(q.s, k), m = scaled(q.m, k), z{0.f, 0.f};
    const df c = o == 0 ? z : (o < 0 ? -q.c : q.c);
    return M22{norm(z2{-(q.w * (v + m)), im}), norm(z2{z, c + s}), norm(z2{z, c - s}), norm(z2{-(q.w * (v - m)), im})};
}

// Number of factor blocks per lane: the cyclic step's pair, a pair per parallel step,
// the even inverse, and the odd nodes' inverse and two couplings.
__host__ __device__ inline int items(int steps) { return 6 + 2 * steps; }

// row h of an item
__device__ __forceinline__ void put(float *tab, int G, int item, int lane, int h, const Row &m) {
    reinterpret_cast<float4 *>(tab + ((size_t)item * G + lane) * 8)[h] = make_float4(m.a.x.h, m.a.y.h, m.b.x.h, m.b.y.h);
}
__device__ __forceinline__ void put_scaled(float *tab, int G, int item, int lane, int h, const Row &m, int k) {   // 2^k m
    reinterpret_cast<float4 *>(tab + ((size_t)item * G + lane) * 8)[h] =
        make_float4(scalbnf(m.a.x.h, k), scalbnf(m.a.y.h, k), scalbnf(m.b.x.h, k), scalbnf(m.b.y.h, k));
}

// The row of one frequency.
__device__ __forceinline__ FreqRow freq_row(const SweepGeom &g, int f) {
    const int i1 = f / g.n2, i2 = f % g.n2;
    double myz, by, bz;
    symbols(g, i1, i2, myz, by, bz);
    const int sys = 2 * (min(i1, g.n1 - i1) * (g.n2 / 2 + 1) + min(i2, g.n2 - i2));
    if (g.nc == 2) return FreqRow{(float)myz, (float)by, 1.f, 0.f, sys + (by < 0.0 ? 1 : 0)};
    const double phi = atan2(bz, by);
    return FreqRow{(float)myz, (float)hypot(by, bz), (float)cos(0.5 * phi), (float)sin(0.5 * phi), sys};
}

// Factors of every distinct system in 48 bits (pairs of floats), stored in FP32: every
// block is scaled by one power of two per system, so that the mass is about 1.  G lanes per
// system; the neighbours' blocks pass through shared memory (three M22 per lane, by
// quarters of 16 bytes, so that a warp's accesses are contiguous).  The CTAs after the last
// system's write the rows of the frequencies.
// Two threads share a lane, a row of every block each: products by rows need nothing of the
// other row, an inverse takes it by a shuffle.
// The 2 x 625 systems of the 48^3 x 48 Klein mesh take 79 us; with whole blocks per thread
// (a chain twice as long on half the warps) 97 us, and in FP64, which kept that unit busy
// throughout, 215 us.
__global__ void __launch_bounds__(512) factor_kernel(SweepGeom g, int G, int steps, const double *__restrict__ Vx,
                                                     float *__restrict__ table, FreqRow *__restrict__ freq) {
    extern __shared__ __align__(16) unsigned char fsm[];
    const int T = blockDim.x / 2, per_cta = T / G;            // nodes and systems of the CTA
    const int fb = (2 * class_count(g.n1, g.n2) + per_cta - 1) / per_cta;
    if ((int)blockIdx.x >= fb) {
        const int f = (blockIdx.x - fb) * blockDim.x + threadIdx.x;
        if (f < g.n1 * g.n2) freq[f] = freq_row(g, f);
        return;
    }
    float4 *xch = reinterpret_cast<float4 *>(fsm);
    const int h = threadIdx.x & 1, node = threadIdx.x / 2, l = node % G, base = node - l;
    const int nsys = 2 * class_count(g.n1, g.n2);
    const int sys = blockIdx.x * per_cta + node / G;
    const bool live = sys < nsys;
    const int cls = (live ? sys : 0) / 2, q2 = g.n2 / 2 + 1;
    double myz, by, bz;
    symbols(g, cls / q2, cls % q2, myz, by, bz);
    const int k2 = -ilogb(myz * g.h[0]);
    myz = scalbn(myz, k2);
    const double P = scalbn(((sys & 1) ? -1.0 : 1.0) * sqrt(by * by + bz * bz), k2), h6 = g.h[0] * (1.0 / 6.0), ht2 = 0.5 * g.ht;
    const BdSymbols q{to_df(h6 * myz), to_df(0.5 * ht2 * myz), to_df(ht2 * h6 * P), to_df(ht2 * h6 * myz), to_df(g.m)};
    const int n = g.nx, e = 2 * l, o = e + 1;
    float *tab = table + (size_t)(live ? sys : 0) * items(steps) * G * 8;
    const df one{1.f, 0.f}, nil{0.f, 0.f};
    const z2 z1{one, nil}, z0{nil, nil};
    const Row none{z0, z0}, unit = h ? Row{z0, z1} : Row{z1, z0};
    Row L = none, U = none, D = unit, Lo = none, Uo = none, Do = unit;
    df v[3];                                                 // elements e, e + 1, e + 2
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = Vx && e + k <= n ? to_df(Vx[e + k]) : nil;
    if (e < n) {
        D = row(bd_block(q, 0, scaled(v[0] + v[1], 2.f)), h);
        if (e > 0) L = row(bd_block(q, -1, v[0]), h);
        if (o < n) {
            U = row(bd_block(q, 1, v[1]), h);
            Do = row(bd_block(q, 0, scaled(v[1] + v[2], 2.f)), h);
            Lo = row(bd_block(q, -1, v[1]), h);
            if (o + 1 < n) Uo = row(bd_block(q, 1, v[2]), h);
        }
    }
    // (both lanes of a node have the same e and o)
    Row Doi = inv_row(Do, h);
    if (o >= n) Doi = none;
    auto put_x = [&](int which, const Row &m) {
        xch[(4 * which + 2 * h) * T + node] = make_float4(m.a.x.h, m.a.x.l, m.a.y.h, m.a.y.l);
        xch[(4 * which + 2 * h + 1) * T + node] = make_float4(m.b.x.h, m.b.x.l, m.b.y.h, m.b.y.l);
    };
    auto get_x = [&](int which, int at) {
        M22 m;
        z2 *z = &m.a;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 w = xch[(4 * which + k) * T + at];
            z[k] = z2{df{w.x, w.y}, df{w.z, w.w}};
        }
        return m;
    };
    auto publish = [&](const Row &a, const Row &b, const Row &c) {
        __syncthreads();
        put_x(0, a); put_x(1, b); put_x(2, c);
        __syncthreads();
    };
    publish(Doi, Lo, Uo);
    {
        const int left = l > 0 ? node - 1 : node;                    // l = 0: L = 0, any block will do
        const M22 Doi2 = get_x(0, node), Lo2 = get_x(1, node), Uo2 = get_x(2, node);
        const Row A = mul(L, get_x(0, left)), Bm = mul(U, Doi2);
        D = sub(sub(D, mul(A, get_x(2, left))), mul(Bm, Lo2));
        L = neg(mul(A, get_x(1, left)));
        U = neg(mul(Bm, Uo2));
        if (live) {
            const int at = 2 + 2 * steps;
            put(tab, G, 0, l, h, A);
            put(tab, G, 1, l, h, Bm);
            put_scaled(tab, G, at + 1, l, h, Doi, k2);
            put(tab, G, at + 2, l, h, mul(Doi, Lo2));
            put(tab, G, at + 3, l, h, mul(Doi, Uo2));
        }
    }
    for (int s = 0; s < steps; ++s) {
        const int st = 1 << s;
        publish(inv_row(D, h), L, U);
        const bool hl = l >= st, hr = l + st < G;
        const int il = hl ? node - st : base, ir = hr ? node + st : base;
        const Row al = hl ? mul(L, get_x(0, il)) : none, ga = hr ? mul(U, get_x(0, ir)) : none;
        D = sub(sub(D, mul(al, get_x(2, il))), mul(ga, get_x(1, ir)));
        L = neg(mul(al, get_x(1, il)));
        U = neg(mul(ga, get_x(2, ir)));
        if (live) { put(tab, G, 2 + 2 * s, l, h, al); put(tab, G, 3 + 2 * s, l, h, ga); }
    }
    const Row Di = inv_row(D, h);
    if (live) put_scaled(tab, G, 2 + 2 * steps, l, h, Di, k2);
}

// hi + lo = 2 sum_t (-1)^t v_t per spatial entry (two complex entries per thread;
// TwoSum keeps the rounding of every addition).
__device__ __forceinline__ void two_add(float &hi, float &lo, float a) {
    const float s = hi + a, bb = s - hi;
    lo += (hi - (s - bb)) + (a - bb);
    hi = s;
}
// s_{t+1} = 2 v_t - s_t
__device__ __forceinline__ void next_s(float4 &s, float4 &lo, const float4 v) {
    s = make_float4(-s.x, -s.y, -s.z, -s.w);
    lo = make_float4(-lo.x, -lo.y, -lo.z, -lo.w);
    two_add(s.x, lo.x, 2.f * v.x); two_add(s.y, lo.y, 2.f * v.y);
    two_add(s.z, lo.z, 2.f * v.z); two_add(s.w, lo.w, 2.f * v.w);
}
__global__ void __launch_bounds__(256) altsum_kernel(int64_t per2, int64_t nt, const float4 *__restrict__ v,
                                                     float4 *__restrict__ hi, float4 *__restrict__ lo) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= per2) return;
    float4 h = make_float4(0.f, 0.f, 0.f, 0.f), r = h;
    constexpr int PD = 8;
    for (int64_t t0 = 0; t0 < nt; t0 += PD) {
        float4 a[PD];
#pragma unroll
        for (int q = 0; q < PD; ++q)
            a[q] = t0 + q < nt ? __ldg(v + (t0 + q) * per2 + e) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < PD; ++q) {
            const float w = (q & 1) ? -2.f : 2.f;
            two_add(h.x, r.x, w * a[q].x); two_add(h.y, r.y, w * a[q].y);
            two_add(h.z, r.z, w * a[q].z); two_add(h.w, r.w, w * a[q].w);
        }
    }
    hi[e] = h;
    lo[e] = r;
}

__device__ __forceinline__ float4 add4(const float4 a, const float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
struct Blk { float4 r0, r1; };            // a 2 x 2 complex block by rows
__device__ __forceinline__ Blk load_blk(const float *tab, int G, int item, int lane) {
    const float4 *o = reinterpret_cast<const float4 *>(tab + ((size_t)item * G + lane) * 8);
    return Blk{__ldg(o), __ldg(o + 1)};
}
// acc += B v, or acc -= B v; v = (v0.re, v0.im, v1.re, v1.im)
__device__ __forceinline__ void add_mv(float4 &acc, const Blk &B, const float4 v) {
    acc.x = fmaf(B.r0.x, v.x, fmaf(-B.r0.y, v.y, fmaf(B.r0.z, v.z, fmaf(-B.r0.w, v.w, acc.x))));
    acc.y = fmaf(B.r0.x, v.y, fmaf(B.r0.y, v.x, fmaf(B.r0.z, v.w, fmaf(B.r0.w, v.z, acc.y))));
    acc.z = fmaf(B.r1.x, v.x, fmaf(-B.r1.y, v.y, fmaf(B.r1.z, v.z, fmaf(-B.r1.w, v.w, acc.z))));
    acc.w = fmaf(B.r1.x, v.y, fmaf(B.r1.y, v.x, fmaf(B.r1.z, v.w, fmaf(B.r1.w, v.z, acc.w))));
}
__device__ __forceinline__ void sub_mv(float4 &acc, const Blk &B, const float4 v) {
    acc.x = fmaf(-B.r0.x, v.x, fmaf(B.r0.y, v.y, fmaf(-B.r0.z, v.z, fmaf(B.r0.w, v.w, acc.x))));
    acc.y = fmaf(-B.r0.x, v.y, fmaf(-B.r0.y, v.x, fmaf(-B.r0.z, v.w, fmaf(-B.r0.w, v.z, acc.y))));
    acc.z = fmaf(-B.r1.x, v.x, fmaf(B.r1.y, v.y, fmaf(-B.r1.z, v.z, fmaf(B.r1.w, v.w, acc.z))));
    acc.w = fmaf(-B.r1.x, v.y, fmaf(-B.r1.y, v.x, fmaf(-B.r1.z, v.w, fmaf(-B.r1.w, v.z, acc.w))));
}

__device__ __forceinline__ void copy16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Shared memory of one CTA of `sys` systems: STAGES input layers, two output layers,
// two exchange buffers of two values per lane.
__host__ __device__ inline int row_bytes(int nc, int sys) { return (nc == 4 ? sys / 2 : sys) * nc * 8 + 16; }
inline size_t march_smem(int nc, int sys, int G, int n) {
    return (size_t)(STAGES + 2) * ((n + 1) / 2 * 2) * row_bytes(nc, sys) + 4 * sizeof(float4) * (size_t)sys * G;
}

// LARGE: h_t K is not small against M (dst_sweep_plan's rule).  The reduction then loses
// digits, so each solve is refined once, on the form Bd x_t = s_t - Bl x_{t-1}.  Below, the
// increment form alone is as exact as an elimination along x in order, or better (relative
// error against FP64 9.3e-7 and 1.5e-6 on the 48^3 x 48 Klein mesh).  With q = h_t (sum of
// 1 / h_k + 2 (m + max |V|)) the error of 48 layers, as a multiple of that elimination's,
// is at most 0.8 unrefined up to q = 1.5 (1+1: 0.9 up to q = 0.6, 1.2 from 0.65 on), 1.2 at 2.3,
// 1.6 at 3.5, 2 to 3.7 from 7 on; refined 0.4 to 0.8 there, 0.5 on average over 338 meshes from
// q = 4 on, above 1.1 in eleven of them (high potentials on short transverse spacings, 1.8
// at most).  A step's refinement takes about as long as its solve: 48^3 x 12 layers 348 us,
// 314 without; 1+1 39 nodes x 40 layers 109 us and 95.
// blockDim.x = systems per CTA x G.  Layers t of `in` [t][x][f][c] to `out` (in == out allowed).
template <int NC, int G, bool LARGE>
__global__ void __launch_bounds__(G > 32 ? 512 : 256)
march_kernel(SweepGeom g, int steps, const double *__restrict__ Vx, const float *__restrict__ table,
             const FreqRow *__restrict__ ft, const float4 *__restrict__ alt_hi, const float4 *__restrict__ alt_lo, const float2 *in, float2 *out) {
    extern __shared__ __align__(16) unsigned char msm[];
    constexpr bool REG = G <= 32;
    const int n = g.nx, half = (n + 1) / 2, rows = 2 * half;
    const int64_t nf = (int64_t)g.n1 * g.n2;
    const int nsys = blockDim.x / G, fper = NC == 4 ? nsys / 2 : nsys;
    const int RB = row_bytes(NC, nsys);
    unsigned char *ring = msm, *otile = ring + (size_t)STAGES * rows * RB;
    float4 *xch = reinterpret_cast<float4 *>(otile + (size_t)2 * rows * RB);
    const int l = threadIdx.x % G, sys = threadIdx.x / G;
    const int slot = NC == 4 ? sys / 2 : sys, pair = NC == 4 ? sys & 1 : 0;
    const int64_t f0 = (int64_t)blockIdx.x * fper, f = f0 + slot;
    const FreqRow fq = ft[f < nf ? f : 0];
    const float *tab = table + (size_t)(fq.sys + pair) * items(steps) * G * 8;
    // rows past the last frequency stay zero
    for (int i = threadIdx.x; i < (STAGES + 2) * rows * RB / 16; i += blockDim.x)
        reinterpret_cast<float4 *>(ring)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    // a row of the ring: the CTA's frequencies of one x node, even nodes first, so that
    // the lanes of a warp read consecutive rows.  A thread copies one 16-byte column of
    // rows i0 and i0 + G (n <= 2 G; G is even, so their places lie G/2 rows apart), the
    // same ones of every layer: with a division and a comparison per piece instead, a
    // third of the issue slots went to addresses (386 us against 255 on the 48^3 x 48
    // Klein mesh).
    const int per_row = fper * NC / 2, ch = threadIdx.x % per_row, i0 = threadIdx.x / per_row;
    const bool column = ch < (nf - f0) * (NC / 2);
    const bool copy0 = column && i0 < n, copy1 = column && i0 + G < n;
    auto pos = [&](int i) { return (i & 1) * half + (i >> 1); };
    const int at0 = pos(i0) * RB + ch * 16, at1 = at0 + (G / 2) * RB, tile = rows * RB;
    const int64_t off0 = (i0 * nf + f0) * NC * 8 + ch * 16, off1 = off0 + (int64_t)G * nf * NC * 8,
                  layer = (int64_t)n * nf * NC * 8;
    const char *src = reinterpret_cast<const char *>(in) + off0;
    char *dst = reinterpret_cast<char *>(out) + off0;
    const int64_t nt = g.nt;
    int64_t issued = 0;
    int fill = 0;                                              // layers issued; the ring slot of the next
    auto issue = [&] {
        if (issued < nt) {
            unsigned char *d = ring + fill;
            if (copy0) copy16(d + at0, src);
            if (copy1) copy16(d + at1, src + (off1 - off0));
            src += layer;
        }
        ++issued;
        fill = fill == (STAGES - 1) * tile ? 0 : fill + tile;
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    // the rotated pair of one node from its two (2+1) or four (3+1) components
    const float rc = fq.c, rs = fq.s;
    auto rotate = [&](const float4 a, const float4 b) {       // a = (v0, v1), b = (v2, v3)
        if (pair == 0) return make_float4(rc * a.x - rs * a.w, rc * a.y + rs * a.z, rc * b.z - rs * b.y, rc * b.w + rs * b.x);
        return make_float4(rc * a.z - rs * a.y, rc * a.w + rs * a.x, rc * b.x - rs * b.w, rc * b.y + rs * b.z);
    };
    auto node = [&](const unsigned char *at) {
        const float4 *q = reinterpret_cast<const float4 *>(at);
        return NC == 4 ? rotate(q[0], q[1]) : q[0];
    };
    auto alt = [&](const float4 *v, int i) {
        if (i >= n || f >= nf) return make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 *q = v + (i * nf + f) * (NC / 2);
        return NC == 4 ? rotate(q[0], q[1]) : q[0];
    };
    const int e = 2 * l, o = e + 1;
    const bool he = e < n, ho = o < n;
    // K' = h_t K (LARGE: h_t / 2 K) of a node between elements of potential a and b, its neighbours p and r:
    // component 0 takes i kC (r - p)_1 + i kP (p + 4 c + r)_1 - sum over both elements of
    // (V + m) kW (neighbour + 2 c)_0, component 1 the same with kP and m negated
    const double hk = LARGE ? 0.5 * g.ht : g.ht;
    const float kC = (float)(0.5 * hk) * fq.myz, kW = (float)(hk * g.h[0] / 6.0) * fq.myz;
    const float kP = (float)(hk * g.h[0] / 6.0) * (pair ? -fq.P : fq.P), km = kW * (float)g.m;
    const float kM = LARGE ? (float)(g.h[0] / 6.0) * fq.myz : 0.f;
    float ve[3];                                              // elements e, e + 1, e + 2
#pragma unroll
    for (int k = 0; k < 3; ++k) ve[k] = Vx && e + k <= n ? kW * (float)Vx[e + k] : 0.f;
    Blk A = load_blk(tab, G, 0, l), Bm = load_blk(tab, G, 1, l);
    Blk al[REG ? REG_STEPS : 1], ga[REG ? REG_STEPS : 1];
    constexpr int LOGG = G == 8 ? 3 : (G == 16 ? 4 : 5);
    if (REG) {
#pragma unroll
        for (int s = 0; s < LOGG; ++s)
            if (s < steps) { al[s] = load_blk(tab, G, 2 + 2 * s, l); ga[s] = load_blk(tab, G, 3 + 2 * s, l); }
    }
    const int at = 2 + 2 * steps;
    Blk Di = load_blk(tab, G, at, l), Oi = load_blk(tab, G, at + 1, l), OL = load_blk(tab, G, at + 2, l),
        OU = load_blk(tab, G, at + 3, l);
    float4 se = alt(alt_hi, e), so = alt(alt_hi, o), sel = alt(alt_lo, e), sol = alt(alt_lo, o);
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 xe = z4, xo = z4, xn = z4;                          // x_{t-1} at e, o and e + 2
    int buf = 0;
    float4 *mine = xch + threadIdx.x, *mine2 = mine + 2 * blockDim.x;
    auto sync = [&] { if (G <= 32) __syncwarp(); else __syncthreads(); };
    auto swap_buf = [&] { buf ^= (int)blockDim.x; };
    const int left = l > 0 ? -1 : 0, right = l + 1 < G ? 1 : 0;
    for (int q = 0; q < STAGES - 1; ++q) issue();

    // s - K' x + i kM M' x of a node between elements of potential va and vb (M' the [1,4,1]
    // sum), x at the node and its neighbours p and r
    auto rhs = [&](const float4 s, const float4 slo, const float4 c, const float4 p, const float4 r, float va, float vb,
                   float kM) {
        const float4 S = make_float4(fmaf(4.f, c.x, p.x + r.x), fmaf(4.f, c.y, p.y + r.y), fmaf(4.f, c.z, p.z + r.z),
                                     fmaf(4.f, c.w, p.w + r.w));
        const float4 E = make_float4(r.x - p.x, r.y - p.y, r.z - p.z, r.w - p.w);
        const float4 a = make_float4(fmaf(2.f, c.x, p.x), fmaf(2.f, c.y, p.y), fmaf(2.f, c.z, p.z), fmaf(2.f, c.w, p.w));
        const float4 b = make_float4(fmaf(2.f, c.x, r.x), fmaf(2.f, c.y, r.y), fmaf(2.f, c.z, r.z), fmaf(2.f, c.w, r.w));
        const float pa = va + km, pb = vb + km, ma = va - km, mb = vb - km;
        float4 q = make_float4(s.x + fmaf(kC, E.w, fmaf(kP, S.w, fmaf(pa, a.x, fmaf(pb, b.x, slo.x)))),
                               s.y + fmaf(-kC, E.z, fmaf(-kP, S.z, fmaf(pa, a.y, fmaf(pb, b.y, slo.y)))),
                               s.z + fmaf(kC, E.y, fmaf(-kP, S.y, fmaf(ma, a.z, fmaf(mb, b.z, slo.z)))),
                               s.w + fmaf(-kC, E.x, fmaf(kP, S.x, fmaf(ma, a.w, fmaf(mb, b.w, slo.w)))));
        if (LARGE) {
            q.x = fmaf(-kM, S.y, q.x); q.y = fmaf(kM, S.x, q.y); q.z = fmaf(-kM, S.w, q.z); q.w = fmaf(kM, S.z, q.w);
        }
        return q;
    };
    // the left lane's v and w (v 0 at the wall, where the factor of w is 0)
    auto from_left = [&](const float4 v, const float4 w, float4 &vl, float4 &wl) {
        mine[buf] = v;
        mine2[buf] = w;
        sync();
        vl = l > 0 ? mine[buf + left] : z4;
        wl = mine2[buf + left];
        swap_buf();
    };
    // Bd u = r; un: u at e + 2
    // (rl: the left lane's ro)
    auto solve = [&](float4 re, const float4 ro, const float4 rl, float4 &ue, float4 &uo, float4 &un) {
        sub_mv(re, A, rl);
        sub_mv(re, Bm, ro);
        auto reduce = [&](int st, const Blk &a, const Blk &b) {
            mine[buf] = re;
            sync();
            const float4 vl = mine[buf + (l >= st ? -st : 0)], vr = mine[buf + (l + st < G ? st : 0)];
            sub_mv(re, a, vl);
            sub_mv(re, b, vr);
            swap_buf();
        };
        if (REG) {
#pragma unroll
            for (int s = 0; s < LOGG; ++s)
                if (s < steps) reduce(1 << s, al[s], ga[s]);
        } else {
            for (int s = 0; s < steps; ++s) reduce(1 << s, load_blk(tab, G, 2 + 2 * s, l), load_blk(tab, G, 3 + 2 * s, l));
        }
        ue = uo = z4;
        add_mv(ue, Di, re);
        mine[buf] = ue;
        sync();
        un = l + 1 < G ? mine[buf + right] : z4;
        swap_buf();
        add_mv(uo, Oi, ro);
        sub_mv(uo, OL, ue);
        sub_mv(uo, OU, un);
    };
    // a finished layer from its tile, rotated back
    float bc = 1.f, bs = 0.f;
    if (NC == 4 && column) { bc = ft[f0 + (ch >> 1)].c; bs = ft[f0 + (ch >> 1)].s; }
    auto store_layer = [&](const unsigned char *t) {
        auto back = [&](const unsigned char *q) {
            const float4 v = *reinterpret_cast<const float4 *>(q);
            if (NC == 2) return v;
            return make_float4(bc * v.x + bs * v.w, bc * v.y - bs * v.z, bc * v.z + bs * v.y, bc * v.w - bs * v.x);
        };
        if (copy0) *reinterpret_cast<float4 *>(dst) = back(t + at0);
        if (copy1) *reinterpret_cast<float4 *>(dst + (off1 - off0)) = back(t + at1);
        dst += layer;
    };
    // this lane's places in a tile
    const int ate = (he ? pos(e) : 0) * RB + slot * NC * 8, ato = (ho ? pos(o) : 0) * RB + slot * NC * 8;
    int used = 0;                                              // the ring slot of layer t
    for (int64_t t = 0; t < nt; ++t) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(STAGES - 2) : "memory");
        __syncthreads();               // layer t staged; layer t - 1 of the output complete; its input slot free
        issue();
        if (t > 0) store_layer(otile + (t & 1 ? 0 : tile));
        // the odd node's right-hand side needs no neighbour beyond e and e + 2, the even one's
        // the left lane's x_{t-1}, which comes with that lane's odd right-hand side: one exchange
        float4 ro = rhs(so, sol, xo, xe, xn, ve[1], ve[2], kM);
        if (!ho) ro = z4;
        float4 xl, rl;
        from_left(xo, ro, xl, rl);
        float4 re = rhs(se, sel, xe, xl, xo, ve[0], ve[1], kM);
        if (!he) re = z4;
        float4 ue, uo, un;
        solve(re, ro, rl, ue, uo, un);
        if (LARGE) {
            // one step of refinement: u += Bd^-1 (r - Bd u)
            ro = rhs(ro, z4, uo, ue, un, ve[1], ve[2], -kM);
            if (!ho) ro = z4;
            from_left(uo, ro, xl, rl);
            re = rhs(re, z4, ue, xl, uo, ve[0], ve[1], -kM);
            if (!he) re = z4;
            float4 de, dd, dn;
            solve(re, ro, rl, de, dd, dn);
            xe = add4(ue, de); xo = add4(uo, dd); xn = add4(un, dn);
        } else {
            xe = add4(ue, xe); xo = add4(uo, xo); xn = add4(un, xn);
        }
        unsigned char *ot = otile + (t & 1 ? tile : 0);
        auto emit = [&](int at, const float4 x) {
            unsigned char *d = ot + at;
            if (NC == 4) {
                *reinterpret_cast<float2 *>(d + (pair ? 8 : 0)) = make_float2(x.x, x.y);
                *reinterpret_cast<float2 *>(d + (pair ? 16 : 24)) = make_float2(x.z, x.w);
            } else {
                *reinterpret_cast<float4 *>(d) = x;
            }
        };
        const unsigned char *it = ring + used;
        used = used == (STAGES - 1) * tile ? 0 : used + tile;
        if (he) { emit(ate, xe); next_s(se, sel, node(it + ate)); }
        if (ho) { emit(ato, xo); next_s(so, sol, node(it + ato)); }
    }
    __syncthreads();
    store_layer(otile + (nt & 1 ? 0 : tile));
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

}  // namespace dst_march
