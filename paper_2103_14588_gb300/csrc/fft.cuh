// FFT of the planes of periodic axes in shared memory (used by the
// Crank-Nicolson sweep in FP32 and by the energy observable in FP64).
//
// Each CTA loads one plane (n1 x n2 nodes of one layer, or of one x node of a
// layer) of its component group into shared memory, transforms every line of
// the inner axis and then every line of the outer axis, and stores the result.
// Mixed-radix Stockham self-sorting stages (16, 8, 4, 2, 3, 5 in registers, other
// primes by their sums; twiddles from a per-axis table w[j] = exp(sign 2 pi i j / n)) run
// either over all lines of an axis at once, the CTA's threads sharing every
// stage's butterflies (when a second plane buffer fits in shared memory), or one
// line per warp with two scratch lines.
// What bounds it is shared memory: with the first and last pass a 48 x 48 plane
// crosses it six times.  Neighbouring lanes take neighbouring lines, whose pitch is
// odd, so that neither the strided reads nor the scattered writes of a stage meet on a
// bank, and the stage's index arithmetic is the same for a whole warp.
// Forward (sign -1): node layout in, frequency layout [b][f][c] out with
// f = i1 n2 + i2.  Inverse (sign +1): frequency layout in, node layout out,
// scaled by 1 / (n1 n2).
#pragma once

#include <algorithm>
#include <type_traits>

#include "sweep.h"

namespace dst_fft {

constexpr int FFT_THREADS = 256;          // at most

template <typename V> struct Real;
template <> struct Real<float2> { using type = float; };
template <> struct Real<double2> { using type = double; };

template <typename V> __device__ __forceinline__ V mk(typename Real<V>::type a, typename Real<V>::type b) {
    V r; r.x = a; r.y = b; return r;
}
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
    return mk<V>(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
template <typename V> __device__ __forceinline__ V cadd(V a, V b) { return mk<V>(a.x + b.x, a.y + b.y); }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { return mk<V>(a.x - b.x, a.y - b.y); }
template <typename V> __device__ __forceinline__ V cfma(V a, V b, V acc) {
    return mk<V>(fma(a.x, b.x, fma(-a.y, b.y, acc.x)), fma(a.x, b.y, fma(a.y, b.x, acc.y)));
}
// a times sg i
template <typename V, typename R> __device__ __forceinline__ V rot(V a, R sg) { return mk<V>(-sg * a.y, sg * a.x); }

__device__ __forceinline__ void sincos_pi(float x, float *s, float *c) { sincospif(x, s, c); }
__device__ __forceinline__ void sincos_pi(double x, double *s, double *c) { sincospi(x, s, c); }

template <int BYTES> __device__ __forceinline__ void copy_async(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(BYTES) : "memory");
}

// Components per CTA, at most (choose_layout).
template <typename V> constexpr int COMPONENTS = sizeof(typename Real<V>::type) == 4 ? 2 : 1;

// What a thread transforms at a time: W components of a node, which lie side by side in
// memory and share index arithmetic, twiddles and wide accesses.
template <typename V, int W> struct alignas(sizeof(V) * W > 16 ? 16 : sizeof(V) * W) Elem { V c[W]; };
template <typename V, int W> __device__ __forceinline__ void copy_elem(Elem<V, W> *dst, const V *src) {
    constexpr int B = (int)sizeof(V) * W;
    if constexpr (B <= 16) copy_async<B>(dst, src);
    else {
        copy_async<16>(dst, src);
        copy_async<16>(reinterpret_cast<char *>(dst) + 16, reinterpret_cast<const char *>(src) + 16);
    }
}

// In-place DFTs of R values, X_o = sum_r v_r exp(sg 2 pi i r o / R).
template <int R> struct Dft;
template <> struct Dft<2> {
    template <typename V, typename S> static __device__ __forceinline__ void run(V *v, S) {
        const V a = v[0], b = v[1];
        v[0] = cadd(a, b); v[1] = csub(a, b);
    }
};
template <> struct Dft<3> {
    template <typename V, typename S> static __device__ __forceinline__ void run(V *v, S sg) {
        const S h = (S)0.86602540378443864676;             // sin(pi / 3)
        const V t = cadd(v[1], v[2]), u = rot(csub(v[1], v[2]), sg * h);
        const V m = mk<V>(fma((S)-0.5, t.x, v[0].x), fma((S)-0.5, t.y, v[0].y));
        v[0] = cadd(v[0], t); v[1] = cadd(m, u); v[2] = csub(m, u);
    }
};
template <> struct Dft<4> {
    template <typename V, typename S> static __device__ __forceinline__ void run(V *v, S sg) {
        const V t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]), t2 = cadd(v[1], v[3]), t3 = rot(csub(v[1], v[3]), sg);
        v[0] = cadd(t0, t2); v[1] = cadd(t1, t3); v[2] = csub(t0, t2); v[3] = csub(t1, t3);
    }
};
template <> struct Dft<5> {
    template <typename V, typename S> static __device__ __forceinline__ void run(V *v, S sg) {
        const S c1 = (S)0.30901699437494742410, c2 = (S)-0.80901699437494742410;     // cos(2 pi / 5), cos(4 pi / 5)
        const S s1 = (S)0.95105651629515357212, s2 = (S)0.58778525229247312917;      // sin(2 pi / 5), sin(4 pi / 5)
        const V a = cadd(v[1], v[4]), b = cadd(v[2], v[3]), d = csub(v[1], v[4]), e = csub(v[2], v[3]);
        const V p = mk<V>(v[0].x + c1 * a.x + c2 * b.x, v[0].y + c1 * a.y + c2 * b.y);
        const V q = mk<V>(v[0].x + c2 * a.x + c1 * b.x, v[0].y + c2 * a.y + c1 * b.y);
        const V r = rot(mk<V>(s1 * d.x + s2 * e.x, s1 * d.y + s2 * e.y), sg);
        const V t = rot(mk<V>(s2 * d.x - s1 * e.x, s2 * d.y - s1 * e.y), sg);
        v[0] = cadd(v[0], cadd(a, b));
        v[1] = cadd(p, r); v[4] = csub(p, r); v[2] = cadd(q, t); v[3] = csub(q, t);
    }
};
template <> struct Dft<8> {
    template <typename V, typename S> static __device__ __forceinline__ void run(V *v, S sg) {
        const S c = (S)0.70710678118654752440;
        V e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        Dft<4>::run(e, sg);
        Dft<4>::run(o, sg);
        o[1] = mk<V>(c * (o[1].x - sg * o[1].y), c * (o[1].y + sg * o[1].x));
        o[2] = rot(o[2], sg);
        o[3] = mk<V>(-c * (o[3].x + sg * o[3].y), c * (sg * o[3].x - o[3].y));
#pragma unroll
        for (int k = 0; k < 4; ++k) { v[k] = cadd(e[k], o[k]); v[k + 4] = csub(e[k], o[k]); }
    }
};
template <> struct Dft<16> {
    template <typename V, typename S> static __device__ __forceinline__ void run(V *v, S sg) {
        const S co[8] = {(S)1, (S)0.92387953251128675613, (S)0.70710678118654752440, (S)0.38268343236508977173,
                         (S)0, (S)-0.38268343236508977173, (S)-0.70710678118654752440, (S)-0.92387953251128675613};
        V e[8], o[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) { e[k] = v[2 * k]; o[k] = v[2 * k + 1]; }
        Dft<8>::run(e, sg);
        Dft<8>::run(o, sg);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const S sn = k == 0 ? (S)0 : (k <= 4 ? co[4 - k] : co[k - 4]);           // sin(pi k / 8)
            const V t = k == 0 ? o[0] : (k == 4 ? rot(o[4], sg) : cmul(o[k], mk<V>(co[k], sg * sn)));
            v[k] = cadd(e[k], t); v[k + 8] = csub(e[k], t);
        }
    }
};

// One butterfly of a stage: elements j + r q of a line (element stride st) times
// w^(r k step), to (j / Ns) Ns R + k + o Ns of the output line; q = n / R, step = q / Ns.
// The first stage (Ns = 1) has no factors.
template <int R, bool FIRST, typename V, int W, typename S>
__device__ __forceinline__ void butterfly(const Elem<V, W> *src, Elem<V, W> *dst, int st, int q, int step, int Ns, int j,
                                          int k, const V *w, S sg) {
    V v[W][R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const Elem<V, W> e = src[(j + r * q) * st];
        const V t = r && !FIRST ? w[r * k * step] : V{};
#pragma unroll
        for (int c = 0; c < W; ++c) v[c][r] = r && !FIRST ? cmul(e.c[c], t) : e.c[c];
    }
#pragma unroll
    for (int c = 0; c < W; ++c) Dft<R>::run(v[c], sg);
    const int to = (j - k) * R + k;
#pragma unroll
    for (int o = 0; o < R; ++o) {
        Elem<V, W> e;
#pragma unroll
        for (int c = 0; c < W; ++c) e.c[c] = v[c][o];
        dst[(to + o * Ns) * st] = e;
    }
}

// One output of a stage of any radix R: V_o = sum_r v_r w^(r (k step + o q)).
template <typename V, int W>
__device__ __forceinline__ Elem<V, W> general_output(const Elem<V, W> *src, int st, int n, int R, int q, int step, int j,
                                                     int k, int o, const V *w) {
    const int inc = k * step + o * q;                      // < n
    Elem<V, W> acc = src[j * st];
    int at = inc;
    for (int r = 1; r < R; ++r) {
        const Elem<V, W> e = src[(j + r * q) * st];
        const V t = w[at];
#pragma unroll
        for (int c = 0; c < W; ++c) acc.c[c] = cfma(t, e.c[c], acc.c[c]);
        at += inc;
        if (at >= n) at -= n;
    }
    return acc;
}

// Every butterfly of one stage for threads `id` of `count`; line l starts at line(l),
// `nl` lines, element stride st; neighbouring threads take neighbouring lines.
template <bool FIRST, typename V, int W, typename S, typename Line>
__device__ __forceinline__ void stage(const Elem<V, W> *d0, Elem<V, W> *d1, int n, int st, int nl, Line line, int R, int Ns,
                                      const V *w, S sg, int id, int count) {
    const int q = n / R, step = q / Ns;
    // quotients by nl and Ns by multiplication: the dividends stay below 2^32 / divisor
    const unsigned rn = nl > 1 ? 0xffffffffu / (unsigned)nl + 1u : 0u, rk = Ns > 1 ? 0xffffffffu / (unsigned)Ns + 1u : 0u;
    auto by_nl = [&](int i) { return nl > 1 ? (int)__umulhi((unsigned)i, rn) : i; };
    auto mod_ns = [&](int j) { return !FIRST && Ns > 1 ? j - (int)__umulhi((unsigned)j, rk) * Ns : 0; };
    auto each = [&](auto radix) {
        constexpr int RR = decltype(radix)::value;
        for (int i = id; i < nl * q; i += count) {
            const int j = by_nl(i), l = i - j * nl, base = line(l), k = mod_ns(j);
            butterfly<RR, FIRST>(d0 + base, d1 + base, st, q, step, Ns, j, k, w, sg);
        }
    };
    switch (R) {
        case 2: each(std::integral_constant<int, 2>()); break;
        case 3: each(std::integral_constant<int, 3>()); break;
        case 4: each(std::integral_constant<int, 4>()); break;
        case 5: each(std::integral_constant<int, 5>()); break;
        case 8: each(std::integral_constant<int, 8>()); break;
        case 16: each(std::integral_constant<int, 16>()); break;
        default:
            for (int i = id; i < nl * n; i += count) {
                const int jo = by_nl(i), l = i - jo * nl, base = line(l);
                const int o = jo / q, j = jo - o * q, k = mod_ns(j);
                d1[base + ((j - k) * R + k + o * Ns) * st] = general_output(d0 + base, st, n, R, q, step, j, k, o, w);
            }
    }
}

template <typename V, int W, typename S>
__device__ __forceinline__ void warp_fft_line(Elem<V, W> *line, int st, int n, const int *rad, int nrad, const V *w, S sg, Elem<V, W> *a,
                              Elem<V, W> *b) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < n; i += 32) a[i] = line[i * st];
    __syncwarp();
    Elem<V, W> *d0 = a, *d1 = b;
    int Ns = 1;
    for (int s = 0; s < nrad; ++s) {
        if (s == 0) stage<true>(d0, d1, n, 1, 1, [](int) { return 0; }, rad[s], 1, w, sg, lane, 32);
        else stage<false>(d0, d1, n, 1, 1, [](int) { return 0; }, rad[s], Ns, w, sg, lane, 32);
        __syncwarp();
        Elem<V, W> *t = d0; d0 = d1; d1 = t;
        Ns *= rad[s];
    }
    for (int i = lane; i < n; i += 32) line[i * st] = d0[i];
    __syncwarp();
}

// All lines of one axis of the plane through the stages at once, with a barrier
// between stages (ping-pong between the two plane buffers).  Returns the buffer that
// holds the result.
template <typename V, int W, typename S, typename Line>
__device__ __forceinline__ Elem<V, W> *cta_fft_axis(Elem<V, W> *d0, Elem<V, W> *d1, int n, int st, int nl, Line line, const int *rad,
                                    int nrad, const V *w, S sg) {
    int Ns = 1;
    for (int s = 0; s < nrad; ++s) {
        if (s == 0) stage<true>(d0, d1, n, st, nl, line, rad[s], 1, w, sg, threadIdx.x, blockDim.x);
        else stage<false>(d0, d1, n, st, nl, line, rad[s], Ns, w, sg, threadIdx.x, blockDim.x);
        __syncthreads();
        Elem<V, W> *t = d0; d0 = d1; d1 = t;
        Ns *= rad[s];
    }
    return d0;
}

// Line pitch of a plane in shared memory: odd where two plane buffers are used.
__host__ __device__ inline int pitch(const SweepFft &a) { return a.pingpong ? a.n2 | 1 : a.n2; }

// Shared memory of one CTA: the plane, two twiddle tables, and a second plane or two
// scratch lines per warp.
// Threads per plane: a butterfly of four points or more each.  A line of 96 nodes alone
// in its plane leaves all but one warp of a larger CTA waiting (2+1 sweep of 96 x 96 x 96:
// 449 us with 256 threads, 302 us with 32); planes of 1024 nodes and more want all 256
// (48 x 48: 698 us against 780 us with 128).
inline unsigned fft_threads(const SweepFft &a) {
    return (unsigned)std::min(FFT_THREADS, std::max(32, (a.n1 * a.n2 / 4 + 31) / 32 * 32));
}
template <typename V>
inline size_t fft_smem_bytes(const SweepFft &a) {
    const int nmax = a.n1 > a.n2 ? a.n1 : a.n2;
    const size_t plane = (size_t)a.ncb * a.n1 * pitch(a);
    const size_t scratch = a.pingpong ? plane : (size_t)(fft_threads(a) / 32) * 2 * nmax * a.ncb;
    return sizeof(V) * (plane + a.n1 + a.n2 + scratch);
}

// W = a.ncb components per CTA.  The direction is a constant of the kernel: the
// multiplications by +-i in the butterflies are then signs of their sums.
template <typename V, int W, bool INVERSE>
__global__ void __launch_bounds__(FFT_THREADS)
fft_planes_kernel(SweepFft a, int64_t ctas, const V *__restrict__ in, V *__restrict__ out) {
    const int64_t cta = blockIdx.y * (int64_t)gridDim.x + blockIdx.x;
    if (cta >= ctas) return;
    using R = typename Real<V>::type;
    constexpr bool inverse = INVERSE;
    constexpr R sign = INVERSE ? (R)1 : (R)-1;
    using E = Elem<V, W>;
    extern __shared__ __align__(16) unsigned char fft_sm_raw[];
    const int n1 = a.n1, n2 = a.n2, nc = a.nc, pt = pitch(a);
    const int nf = n1 * n2, pl = n1 * pt, nmax = n1 > n2 ? n1 : n2;
    E *plane = reinterpret_cast<E *>(fft_sm_raw);         // [n1][pitch]
    E *scr = plane + pl;                                  // second plane, or per warp two lines of nmax
    V *w1 = reinterpret_cast<V *>(scr + (a.pingpong ? pl : (int)(blockDim.x >> 5) * 2 * nmax));   // twiddles of the outer axis (n1)
    V *w2 = w1 + n1;                                      // twiddles of the inner axis (n2)
    // the component groups of a plane are neighbours in the grid: together they use the
    // sectors that each touches half of (apart, DRAM saw three times the plane's bytes)
    const int groups = nc / W;
    const int64_t b = cta / groups;
    const int c0 = (int)(cta - b * groups) * W;
    const int64_t base = (b / a.nbx) * a.ns_nodes + (b % a.nbx) * a.sbx;   // node index of (i1, i2) = (0, 0)
    const unsigned r2 = n2 > 1 ? 0xffffffffu / (unsigned)n2 + 1u : 0u;
    auto row = [&](int f) { return n2 > 1 ? (int)__umulhi((unsigned)f, r2) : f; };
    const V *src = in + (inverse ? b * nf : base) * nc + c0;
#pragma unroll 4
    for (int f = threadIdx.x; f < nf; f += blockDim.x) {
        const int i1 = row(f), i2 = f - i1 * n2;
        copy_elem<V, W>(plane + i1 * pt + i2, src + (inverse ? (int64_t)f : i1 * a.s1 + i2 * a.s2) * nc);
    }
    // the twiddles while the plane is on its way
    for (int j = threadIdx.x; j < n1 && a.nrad1 > 0; j += blockDim.x) {
        R sn, cs;
        sincos_pi((R)2 * (R)j / (R)n1, &sn, &cs);
        w1[j] = mk<V>(cs, sign * sn);
    }
    for (int j = threadIdx.x; j < n2 && a.nrad2 > 0; j += blockDim.x) {
        R sn, cs;
        sincos_pi((R)2 * (R)j / (R)n2, &sn, &cs);
        w2[j] = mk<V>(cs, sign * sn);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    E *cur = plane;
    if (a.pingpong) {
        // CTA-wide stages; scr is a second plane.  Inner lines start every pitch, outer line i2 at i2.
        if (n2 > 1) cur = cta_fft_axis(cur, scr, n2, 1, n1, [&](int l) { return l * pt; }, a.rad2, a.nrad2, w2, sign);
        if (n1 > 1)
            cur = cta_fft_axis(cur, cur == plane ? scr : plane, n1, pt, n2, [](int l) { return l; }, a.rad1, a.nrad1, w1, sign);
    } else {
        const int warp = threadIdx.x >> 5;
        E *sa = scr + (size_t)warp * 2 * nmax, *sb = sa + nmax;
        if (n2 > 1)
            for (int line = warp; line < n1; line += blockDim.x >> 5)
                warp_fft_line(plane + (size_t)line * n2, 1, n2, a.rad2, a.nrad2, w2, sign, sa, sb);
        __syncthreads();
        if (n1 > 1)
            for (int line = warp; line < n2; line += blockDim.x >> 5)
                warp_fft_line(plane + line, n2, n1, a.rad1, a.nrad1, w1, sign, sa, sb);
        __syncthreads();
    }
    const R scale = inverse ? (R)1 / (R)nf : (R)1;
    V *dst = out + (inverse ? base : b * nf) * nc + c0;
    for (int f = threadIdx.x; f < nf; f += blockDim.x) {
        const int i1 = row(f), i2 = f - i1 * n2;
        E v = cur[i1 * pt + i2];
#pragma unroll
        for (int c = 0; c < W; ++c) { v.c[c].x *= scale; v.c[c].y *= scale; }
        *reinterpret_cast<E *>(dst + (inverse ? i1 * a.s1 + i2 * a.s2 : (int64_t)f) * nc) = v;
    }
}

// The planes `nb` of every component group.  The kernel's shared-memory limit is a
// per-device attribute, set once.
template <typename V, bool INVERSE>
inline cudaError_t fft_launch(const SweepFft &a, int64_t nb, const V *in, V *out, cudaStream_t s) {
    static bool configured[64] = {};
    const auto one = fft_planes_kernel<V, 1, INVERSE>, two = fft_planes_kernel<V, COMPONENTS<V>, INVERSE>;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !configured[dev]) {
        const int limit = 200 * 1024;
        e = cudaFuncSetAttribute(one, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(two, cudaFuncAttributeMaxDynamicSharedMemorySize, limit);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) configured[dev] = true;
    }
    // a caller's FP32 vector may start at any entry (8 bytes): then one component at a time
    SweepFft b = a;
    if ((((uintptr_t)in | (uintptr_t)out) & 15) != 0) b.ncb = 1;
    // (more CTAs than a grid's x extent takes go on in y)
    const int64_t ctas = nb * (b.nc / b.ncb), row = std::min<int64_t>(ctas, 1 << 30);
    const dim3 grid((unsigned)row, (unsigned)((ctas + row - 1) / row));
    (b.ncb == 2 ? two : one)<<<grid, fft_threads(b), fft_smem_bytes<V>(b), s>>>(b, ctas, in, out);
    return cudaGetLastError();
}

// Pick the components per CTA and the stage layout for planes of a.n1 x a.n2:
// CTA-wide stages (second plane buffer) when they fit, else one line per warp; two
// components per CTA in FP32, where they share index arithmetic and twiddles, where three
// such CTAs fit an SM (76 KB; 48 x 48 planes of Klein 48^4: 727 us the sweep, 799 one by
// one) and there are two for every SM (nb planes per component group; from 1 to 1216 CTAs
// no mesh below a few microseconds' difference).  FP64 takes one: its stages wait for the FP64 unit,
// and more lanes with less work each suit it better (energy of 32 x 32 x 400: 157 us, 187 by twos).
// Returns false if nothing fits in `limit` bytes.
template <typename V>
inline bool choose_layout(SweepFft &a, int64_t nb, size_t limit) {
    for (int pp = 1; pp >= 0; --pp) {
        a.pingpong = pp;
        a.ncb = COMPONENTS<V>;                 // spinors have two or four components
        if (a.ncb > 1 && fft_smem_bytes<V>(a) <= (pp ? std::min<size_t>(limit, 76 * 1024) : limit) && nb * (a.nc / 2) >= 304)
            return true;
        a.ncb = 1;
        if (fft_smem_bytes<V>(a) <= limit) return true;
    }
    return false;
}

// Stockham radices of n: the fewest stages of the register butterflies, then other primes.
// `points` (FP64): nodes of the plane; radices of 8 and 16 then want 128 butterflies, four full
// warps, because an FP64 instruction takes its unit's 64 clocks whatever lanes it serves
// (energy of 16 x 16 x 16: 49 us, 55 with one stage of 16 per axis; 1+1 512 x 2000 299 us, 323).
inline void radices(int n, int *r, int &nr, int64_t points = 1 << 30) {
    nr = 0;
    for (int p : {16, 8, 4, 2, 3, 5})
        while (n % p == 0 && (p < 8 || points / p >= 128)) { r[nr++] = p; n /= p; }
    for (int p = 7; n > 1; p += 2)
        while (n % p == 0) { r[nr++] = p; n /= p; }
}

}  // namespace dst_fft
