// Operator apply and right-hand side instantiated for 2+1 dimensions (NC = 2).
// Large meshes without an open axis and with an x-only or no potential take the tiled
// kernel of apply_pipe.cuh, in FP32 its two-threads-per-node form (apply_pipe2h.cuh); the
// others apply_node.cuh.
#include "apply_pipe2h.cuh"

int dst_launch_apply_d2(const OpParams &p, int precision, const void *x, void *y, cudaStream_t s) {
    const bool tiles = dst::tiles_pay<2>(p);
    if (precision == DST_FP64) {
        if (tiles) return dst::launch_apply_pipe<2, 2, double>(p, (const double2 *)x, (double2 *)y, s);
        return dst::launch_apply_node<2, 2, double>(p, (const double2 *)x, (double2 *)y, s);
    }
    if (tiles) {
        const int tv = p.tile_variant[DST_FP32];
        if (tv == 1) return dst::launch_apply_pipe2h<1>(p, (const float2 *)x, (float2 *)y, s);
        if (tv == 2) return dst::launch_apply_pipe2h<2>(p, (const float2 *)x, (float2 *)y, s);
        return dst::launch_apply_pipe2h<0>(p, (const float2 *)x, (float2 *)y, s);
    }
    return dst::launch_apply_node<2, 2, float>(p, (const float2 *)x, (float2 *)y, s);
}

int dst_launch_rhs_d2(const OpParams &p, const double2 *psi0, double2 *b, cudaStream_t s) {
    return dst::launch_rhs<2, 2>(p, psi0, b, s);
}
