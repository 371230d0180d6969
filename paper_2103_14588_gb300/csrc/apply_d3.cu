// Operator apply and right-hand side instantiated for 3+1 dimensions (NC = 4).
// Large meshes without an open axis and with an x-only or no potential take the tiled
// kernel of apply_pipe.cuh or the z-column kernel of apply_zblk.cuh (tile variant 1);
// the others apply_node.cuh.
#include "apply_zblk.cuh"

int dst_launch_apply_d3(const OpParams &p, int precision, const void *x, void *y, cudaStream_t s) {
    const bool tiles = dst::tiles_pay<3>(p);
    if (precision == DST_FP64) {
        // the tiled FP64 kernels save work only where their tiles are many: 24^4 341 us here,
        // 533 tiled; 48^4 4.89 and 4.79 ms
        if (tiles && p.ax[0].n * p.ax[1].n * p.ax[2].n * p.nt >= 1 << 20)
            return dst::launch_apply_pipe<3, 4, double>(p, (const double2 *)x, (double2 *)y, s);
        return dst::launch_apply_node<3, 4, double>(p, (const double2 *)x, (double2 *)y, s);
    }
    if (tiles) return dst::launch_apply_pipe<3, 4, float>(p, (const float2 *)x, (float2 *)y, s);
    return dst::launch_apply_node<3, 4, float>(p, (const float2 *)x, (float2 *)y, s);
}

int dst_launch_rhs_d3(const OpParams &p, const double2 *psi0, double2 *b, cudaStream_t s) {
    return dst::launch_rhs<3, 4>(p, psi0, b, s);
}
