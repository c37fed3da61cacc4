// pf_stage_s32k0.cu -- slot-storage instantiations of the FP32 stage passes (K = 0).
#include "pf_internal.h"

namespace pfk {

int launch_s32k0(const Geom &g, const Pass<float> &P, unsigned sig, cudaStream_t st, const float *A,
             const float *B, const float *L, const signed char *ptype, bool *done)
{
    const dim3 grid(g.tiles_x, g.tiles_y, g.nz);
    *done = true;
    if (g.dim == 2 && sig == (SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 2 && sig == (SIG_P2 | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_P2 | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_P2 | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 2 && sig == (SIG_P0 | SIG_P2 | SIG_R0IN | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_P0 | SIG_P2 | SIG_R0IN | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_P0 | SIG_P2 | SIG_R0IN | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 2 && sig == (SIG_R0OUT | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_R0OUT | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_R0OUT | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 2 && sig == (SIG_ERR)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_ERR, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_ERR, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 2 && sig == (SIG_P0 | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_P0 | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_P0 | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 2 && sig == (SIG_RHS)) {
        if (g.uni) launch_pass(slot_kernel<2, 0, SIG_RHS, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<2, 0, SIG_RHS, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_P2 | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_P2 | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_P2 | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_P0 | SIG_P2 | SIG_R0IN | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_P0 | SIG_P2 | SIG_R0IN | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_P0 | SIG_P2 | SIG_R0IN | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_R0OUT | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_R0OUT | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_R0OUT | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_ERR)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_ERR, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_ERR, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_P0 | SIG_PROJECT)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_P0 | SIG_PROJECT, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_P0 | SIG_PROJECT, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    if (g.dim == 3 && sig == (SIG_RHS)) {
        if (g.uni) launch_pass(slot_kernel<3, 0, SIG_RHS, true>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        else launch_pass(slot_kernel<3, 0, SIG_RHS, false>, grid, BLOCK, 0, st, g, P, A, B, L, ptype);
        return (int)cudaGetLastError();
    }
    *done = false;
    return 0;
}

}  // namespace pfk
