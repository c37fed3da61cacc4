// pf_internal.h -- declarations shared by the engine's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include "pf_kernels.cuh"
#include "pf_vec.cuh"
#include "pf_dbl.cuh"
#include "pf_slots.cuh"

namespace pfk {

// Launches a pass kernel so that it may start while the kernel before it on the
// stream drains (every kernel launched so begins with pass_begin, which waits
// for that kernel's results).  The gap between two dependent kernels is about
// 1.5 us of a pass of 4 to 6 us at the grids of the 2D benchmarks: 128^2 circle,
// RKL2, 20 attempts 3.63 -> 2.77 ms, 1024 x 256 strip 3.68 -> 3.20 ms, 24 batched
// problems 9.84 -> 8.79 ms; large grids gain the drain of the last wave.
template <typename... KA, typename... A>
inline void launch_pass(void (*kernel)(KA...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, const A &...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}

// Launch one fused pass: the instantiation is chosen from the pass signature
// (specialised FP32 hot passes) or the generic kernel.  Returns a cudaError_t.
// tma: tensor maps of the pass's buffers for the TMA-staged FP32 kernels
// (nullptr: plain loads).
// *nk (may be null) receives the number of kernels the pass launched, *kept
// (may be null) whether it wrote the segment words of its output vectors.
template <typename T>
int launch_stage(const Geom &g, const Pass<T> &P, cudaStream_t st, const T *A, const T *B, const T *L,
                 const signed char *ptype, const TmaMaps *tma, int *nk = nullptr, bool *kept = nullptr);

// Kernels one pass of the device-driven loop launches (two-cell passes add
// the wide pass of their crowded cells).
template <typename T>
int kernels_per_pass_d(const Geom &g);

// Launch one pass whose description (buffers, coefficients) sits in device
// memory at dP, written there by a planning kernel before the launch runs
// (device-driven adaptive steps).  sig: the pass signature the description
// will have (stage 1, RKL body or error sweep).  Returns a cudaError_t.
template <typename T>
int launch_stage_d(const Geom &g, unsigned sig, const Pass<T> *dP, cudaStream_t st, const T *A, const T *B,
                   const T *L, const signed char *ptype);

// Packed launch of one pass kind (dimension dim, K, signature sig) over the n
// problems of a device table (two-cell FP32 passes; see VecInst): blocks is
// the sum of their block counts, bstart their prefix sums, crowds whether any
// of them can have crowded cells (vec_crowds), done a zeroed device counter of
// the caller.  Returns a cudaError_t; *ok false when the
// pass kind has no packed form.
int launch_packed(int dim, int K, unsigned sig, const VecInst *tab, const int *bstart, int n, int blocks, bool crowds,
                  int *done, cudaStream_t st, bool *ok);

// Opt every instantiation into its shared memory on the current device;
// returns the resident blocks per SM of the generic 3D kernel (<= 0: error).
template <typename T>
int prepare_stage();

}  // namespace pfk
