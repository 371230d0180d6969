// Streaming operator apply for potentials that depend on x only (or vanish).
//
// Same operator and evaluation order as apply_impl.cuh (sum-factorised Q1
// stencils, spatial fields per time plane combined with the spin matrices,
// time stencils through two running accumulators), but organised for
// bandwidth: one thread owns one spatial node and marches through a chunk of
// time planes.  Its spatial
// neighbours come straight from global memory through L1 as 16-byte vector
// loads - every node of a plane is read by up to 3^d threads of the same CTA,
// so L1/L2 absorb the reuse and DRAM sees each x value about once - and
// nothing is staged in shared memory, so there are no barriers.  In FP32 the
// loads of plane p+1 are issued before plane p is combined (software
// pipelining).
#pragma once

#include "apply_impl.cuh"

namespace dst {

template <int NC, typename T>
struct NodeV {
    typename C2<T>::type c[NC];
};

// Vector load of one node's NC complex values (zero when absent).
template <int NC, typename T>
__device__ __forceinline__ void load_node(const typename C2<T>::type *__restrict__ base, int64_t node, bool ok,
                                          NodeV<NC, T> &v) {
    using V = typename C2<T>::type;
    if (!ok) {
#pragma unroll
        for (int c = 0; c < NC; ++c) v.c[c] = cz<V>();
        return;
    }
    const V *p = base + node * NC;
    if (sizeof(T) == 4) {
        const float4 *q = reinterpret_cast<const float4 *>(p);
#pragma unroll
        for (int k = 0; k < NC / 2; ++k) {
            float4 f = __ldg(q + k);
            v.c[2 * k].x = f.x; v.c[2 * k].y = f.y; v.c[2 * k + 1].x = f.z; v.c[2 * k + 1].y = f.w;
        }
    } else {
        const double2 *q = reinterpret_cast<const double2 *>(p);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            double2 f = __ldg(q + c);
            v.c[c].x = f.x; v.c[c].y = f.y;
        }
    }
}

template <int NC, typename T>
__device__ __forceinline__ void store_node(typename C2<T>::type *__restrict__ base, int64_t node,
                                           const typename C2<T>::type *val) {
    using V = typename C2<T>::type;
    V *p = base + node * NC;
    if (sizeof(T) == 4) {
        float4 *q = reinterpret_cast<float4 *>(p);
#pragma unroll
        for (int k = 0; k < NC / 2; ++k)
            q[k] = make_float4(val[2 * k].x, val[2 * k].y, val[2 * k + 1].x, val[2 * k + 1].y);
    } else {
        double2 *q = reinterpret_cast<double2 *>(p);
#pragma unroll
        for (int c = 0; c < NC; ++c) q[c] = make_double2(val[c].x, val[c].y);
    }
}

// G_C, G_M of one output node from its 3^d neighbourhood; get(r) returns the
// node of neighbourhood row r (r = (dz*NY + dy)*3 + dx), from registers or memory.
template <int D, int NC, typename T, typename Get>
__device__ __forceinline__ void fields(Get get, const NodeCoef<D, T> &k, typename C2<T>::type *GC,
                                       typename C2<T>::type *GM) {
    using V = typename C2<T>::type;
    const int NZ = D >= 3 ? 3 : 1, NY = D >= 2 ? 3 : 1;
    V sM[NC], sW[NC], sCx[NC], sCy[NC], sCz[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) { sM[c] = cz<V>(); sW[c] = cz<V>(); sCx[c] = cz<V>(); sCy[c] = cz<V>(); sCz[c] = cz<V>(); }
    // x-direction weights of the mass + potential term for beta = +1 / -1
    T wx[2][3];
#pragma unroll
    for (int sb = 0; sb < 2; ++sb) {
        wx[sb][0] = k.wl[sb] * k.cx.ml[0];
        wx[sb][1] = k.wl[sb] * k.cx.ml[1] + k.wr[sb] * k.cx.mr[1];
        wx[sb][2] = k.wr[sb] * k.cx.mr[2];
    }
#pragma unroll
    for (int dz = 0; dz < NZ; ++dz) {
        V pM[NC], pCx[NC], pCy[NC], pW[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) { pM[c] = cz<V>(); pCx[c] = cz<V>(); pCy[c] = cz<V>(); pW[c] = cz<V>(); }
#pragma unroll
        for (int dy = 0; dy < NY; ++dy) {
            const int r = (dz * NY + dy) * 3;
            const NodeV<NC, T> n0 = get(r), n1 = get(r + 1), n2 = get(r + 2);
            const T my = D >= 2 ? k.cy.m[dy] : (T)1;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int sb = Beta<D>::s(c) > 0 ? 0 : 1;
                const V x0 = n0.c[c], x1 = n1.c[c], x2 = n2.c[c];
                const V rM = cfma_r(k.cx.m[0], x0, cfma_r(k.cx.m[1], x1, cmul_r(k.cx.m[2], x2)));
                const V rC = cfma_r(k.cx.c[0], x0, cfma_r(k.cx.c[1], x1, cmul_r(k.cx.c[2], x2)));
                const V rW = cfma_r(wx[sb][0], x0, cfma_r(wx[sb][1], x1, cmul_r(wx[sb][2], x2)));
                pM[c] = cfma_r(my, rM, pM[c]);
                pCx[c] = cfma_r(my, rC, pCx[c]);
                pW[c] = cfma_r(my, rW, pW[c]);
                if (D >= 2) pCy[c] = cfma_r(k.cy.c[dy], rM, pCy[c]);
            }
        }
        const T mz = D >= 3 ? k.cz.m[dz] : (T)1;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            sM[c] = cfma_r(mz, pM[c], sM[c]);
            sCx[c] = cfma_r(mz, pCx[c], sCx[c]);
            sW[c] = cfma_r(mz, pW[c], sW[c]);
            if (D >= 2) sCy[c] = cfma_r(mz, pCy[c], sCy[c]);
            if (D >= 3) sCz[c] = cfma_r(k.cz.c[dz], pM[c], sCz[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) { GC[c] = cmul_i(sM[c]); GM[c].x = -sW[c].x; GM[c].y = -sW[c].y; }
    V aS[NC];
    alpha_apply<NC>(0, sCx, aS);
#pragma unroll
    for (int c = 0; c < NC; ++c) GM[c] = cadd(GM[c], cmul_i(aS[c]));
    if (D >= 2) {
        alpha_apply<NC>(1, sCy, aS);
#pragma unroll
        for (int c = 0; c < NC; ++c) GM[c] = cadd(GM[c], cmul_i(aS[c]));
    }
    if (D >= 3) {
        alpha_apply<NC>(2, sCz, aS);
#pragma unroll
        for (int c = 0; c < NC; ++c) GM[c] = cadd(GM[c], cmul_i(aS[c]));
    }
}

// fields() for a vanishing potential: the mass term is m beta S_M, so the
// weighted x stencil and its y / z sums are skipped.
template <int D, int NC, typename T, typename Get>
__device__ __forceinline__ void fields_nov(Get get, const NodeCoef<D, T> &k, T m, typename C2<T>::type *GC,
                                           typename C2<T>::type *GM) {
    using V = typename C2<T>::type;
    const int NZ = D >= 3 ? 3 : 1, NY = D >= 2 ? 3 : 1;
    V sM[NC], sCx[NC], sCy[NC], sCz[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) { sM[c] = cz<V>(); sCx[c] = cz<V>(); sCy[c] = cz<V>(); sCz[c] = cz<V>(); }
#pragma unroll
    for (int dz = 0; dz < NZ; ++dz) {
        V pM[NC], pCx[NC], pCy[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) { pM[c] = cz<V>(); pCx[c] = cz<V>(); pCy[c] = cz<V>(); }
#pragma unroll
        for (int dy = 0; dy < NY; ++dy) {
            const int r = (dz * NY + dy) * 3;
            const NodeV<NC, T> n0 = get(r), n1 = get(r + 1), n2 = get(r + 2);
            const T my = D >= 2 ? k.cy.m[dy] : (T)1;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const V x0 = n0.c[c], x1 = n1.c[c], x2 = n2.c[c];
                const V rM = cfma_r(k.cx.m[0], x0, cfma_r(k.cx.m[1], x1, cmul_r(k.cx.m[2], x2)));
                const V rC = cfma_r(k.cx.c[0], x0, cfma_r(k.cx.c[1], x1, cmul_r(k.cx.c[2], x2)));
                pM[c] = cfma_r(my, rM, pM[c]);
                pCx[c] = cfma_r(my, rC, pCx[c]);
                if (D >= 2) pCy[c] = cfma_r(k.cy.c[dy], rM, pCy[c]);
            }
        }
        const T mz = D >= 3 ? k.cz.m[dz] : (T)1;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            sM[c] = cfma_r(mz, pM[c], sM[c]);
            sCx[c] = cfma_r(mz, pCx[c], sCx[c]);
            if (D >= 2) sCy[c] = cfma_r(mz, pCy[c], sCy[c]);
            if (D >= 3) sCz[c] = cfma_r(k.cz.c[dz], pM[c], sCz[c]);
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        GC[c] = cmul_i(sM[c]);
        const T mb = Beta<D>::s(c) > 0 ? -m : m;        // -(m beta)
        GM[c] = cmul_r(mb, sM[c]);
    }
    V aS[NC];
    alpha_apply<NC>(0, sCx, aS);
#pragma unroll
    for (int c = 0; c < NC; ++c) GM[c] = cadd(GM[c], cmul_i(aS[c]));
    if (D >= 2) {
        alpha_apply<NC>(1, sCy, aS);
#pragma unroll
        for (int c = 0; c < NC; ++c) GM[c] = cadd(GM[c], cmul_i(aS[c]));
    }
    if (D >= 3) {
        alpha_apply<NC>(2, sCz, aS);
#pragma unroll
        for (int c = 0; c < NC; ++c) GM[c] = cadd(GM[c], cmul_i(aS[c]));
    }
}

}  // namespace dst
