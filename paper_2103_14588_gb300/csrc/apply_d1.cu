// Operator apply and right-hand side instantiated for 1+1 dimensions (NC = 2).
// Large FP32 meshes without an open axis and with an x-only or no potential take the
// pipelined kernel of apply_pipe.cuh; the others, and FP64 (1024^2 99 us, 149 tiled), apply_node.cuh.
#include "apply_pipe.cuh"

int dst_launch_apply_d1(const OpParams &p, int precision, const void *x, void *y, cudaStream_t s) {
    if (precision == DST_FP64) return dst::launch_apply_node<1, 2, double>(p, (const double2 *)x, (double2 *)y, s);
    if (dst::tiles_pay<1>(p)) return dst::launch_apply_pipe<1, 2, float>(p, (const float2 *)x, (float2 *)y, s);
    return dst::launch_apply_node<1, 2, float>(p, (const float2 *)x, (float2 *)y, s);
}

bool dst_apply_tiled(const OpParams &p, int d) {
    return d == 1 ? dst::tiles_pay<1>(p) : d == 2 ? dst::tiles_pay<2>(p) : dst::tiles_pay<3>(p);
}

int dst_launch_rhs_d1(const OpParams &p, const double2 *psi0, double2 *b, cudaStream_t s) {
    return dst::launch_rhs<1, 2>(p, psi0, b, s);
}
