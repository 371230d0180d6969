// Operator apply and right-hand side instantiated for 3+1 dimensions (NC = 4).
// Large meshes without an open axis and with an x-only or no potential take the column
// kernel of apply_col.cuh, the others apply_node.cuh.
#include "apply_col.cuh"

int dst_launch_apply_d3(const OpParams &p, int precision, const void *x, void *y, cudaStream_t s) {
    const bool tiles = dst::tiles_pay<3>(p);
    if (precision == DST_FP64) {
        if (tiles) return dst::launch_apply_col<double>(p, (const double2 *)x, (double2 *)y, s);
        return dst::launch_apply_node<3, 4, double>(p, (const double2 *)x, (double2 *)y, s);
    }
    if (tiles) return dst::launch_apply_col<float>(p, (const float2 *)x, (float2 *)y, s);
    return dst::launch_apply_node<3, 4, float>(p, (const float2 *)x, (float2 *)y, s);
}

int dst_launch_rhs_d3(const OpParams &p, const double2 *psi0, double2 *b, cudaStream_t s) {
    return dst::launch_rhs<3, 4>(p, psi0, b, s);
}
