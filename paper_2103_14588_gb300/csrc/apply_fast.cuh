// Spatial fields of one node with general stencil coefficients, for the tiles of
// apply_pipe.cuh that meet an open axis (the batched solves; 1+1 and 2+1).
//
// Same operator and evaluation order as apply_impl.cuh: sum-factorised Q1 stencils of a
// time plane, combined with the spin matrices into G_C and G_M.
#pragma once

#include "apply_impl.cuh"

namespace dst {

template <int NC, typename T>
struct NodeV {
    typename C2<T>::type c[NC];
};

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

// G_C, G_M of one output node from its 3^d neighbourhood (d = 1, 2); get(r) returns the
// node of neighbourhood row r (r = dy*3 + dx).
template <int D, int NC, typename T, typename Get>
__device__ __forceinline__ void fields(Get get, const NodeCoef<D, T> &k, typename C2<T>::type *GC,
                                       typename C2<T>::type *GM) {
    using V = typename C2<T>::type;
    const int NY = D >= 2 ? 3 : 1;
    V sM[NC], sW[NC], sCx[NC], sCy[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) { sM[c] = cz<V>(); sW[c] = cz<V>(); sCx[c] = cz<V>(); sCy[c] = cz<V>(); }
    // x-direction weights of the mass + potential term for beta = +1 / -1
    T wx[2][3];
#pragma unroll
    for (int sb = 0; sb < 2; ++sb) {
        wx[sb][0] = k.wl[sb] * k.cx.ml[0];
        wx[sb][1] = k.wl[sb] * k.cx.ml[1] + k.wr[sb] * k.cx.mr[1];
        wx[sb][2] = k.wr[sb] * k.cx.mr[2];
    }
#pragma unroll
    for (int dy = 0; dy < NY; ++dy) {
        const int r = dy * 3;
        const NodeV<NC, T> n0 = get(r), n1 = get(r + 1), n2 = get(r + 2);
        const T my = D >= 2 ? k.cy.m[dy] : (T)1;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int sb = Beta<D>::s(c) > 0 ? 0 : 1;
            const V x0 = n0.c[c], x1 = n1.c[c], x2 = n2.c[c];
            const V rM = cfma_r(k.cx.m[0], x0, cfma_r(k.cx.m[1], x1, cmul_r(k.cx.m[2], x2)));
            const V rC = cfma_r(k.cx.c[0], x0, cfma_r(k.cx.c[1], x1, cmul_r(k.cx.c[2], x2)));
            const V rW = cfma_r(wx[sb][0], x0, cfma_r(wx[sb][1], x1, cmul_r(wx[sb][2], x2)));
            sM[c] = cfma_r(my, rM, sM[c]);
            sCx[c] = cfma_r(my, rC, sCx[c]);
            sW[c] = cfma_r(my, rW, sW[c]);
            if (D >= 2) sCy[c] = cfma_r(k.cy.c[dy], rM, sCy[c]);
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
}

}  // namespace dst
