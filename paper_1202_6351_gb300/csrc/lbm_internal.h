// lbm_internal.h -- host-side declarations shared by the library's translation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "lbm_device.cuh"

struct lbm_s;  // the handle behind lbm_t (lbm_handle.h)

namespace lbm {

// Kernels of one chain of launches overlap their launch with the end of the
// kernel before: the next grid is set up while the last blocks finish, and
// every kernel launched this way calls pdl_wait, which returns when the grid
// before has completed and its writes are visible, before it touches global
// memory.  Its pointer arguments are not __restrict__: the memory is written by
// others while it waits.  No kernel asks for the next one earlier (launch_dependents): blocks
// placed while the current grid still holds most slots end up unevenly spread
// over the SMs (FP32 257^2: 2.35 us per step so, 1.92 without; 2.16 without any
// overlap).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_chain(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

// 0: no force, 1: uniform force only, 2: per-node field (plus the uniform force).
int force_mode(const lbm_s* h);

// One fused step of any storage kind on the population array a.f.
cudaError_t launch_step_any(const Args& a, int store, int model, bool odd, int force, bool walls, cudaStream_t s);

// Launch shape of the fused step kernel: one thread per node, BX x BY threads.
// Blocks of 128 threads rather than 256 leave a shorter last wave and spread more
// evenly: FP32 us per step 512^2 3.17 -> 3.13, cavity 512^2 3.55 -> 3.38, 257^2 1.92 ->
// 1.70, 1025^2 9.35 -> 9.09, 4096^2 189.6 -> 184.1 (384^2 2.15 -> 2.21); 64 threads are
// slower from 384^2 to 1025^2.
constexpr int kStepBX = 128;
constexpr int kStepBY = 1;

// One fused collide-and-stream step (defined once per storage type).
cudaError_t launch_step_f64(const Args& a, int model, bool odd, int force, bool walls, cudaStream_t s);
cudaError_t launch_step_f32(const Args& a, int model, bool odd, int force, bool walls, cudaStream_t s);
cudaError_t launch_step_bf16(const Args& a, int model, bool odd, int force, bool walls, cudaStream_t s);
cudaError_t launch_step_f16(const Args& a, int model, bool odd, int force, bool walls, cudaStream_t s);

// Two fused steps (variant 3, lbm_fused.cuh) from a.f (natural layout, even
// step) into `out`; `map` describes a.f.  FP32, BF16 and FP16 storage.
cudaError_t launch_fused_f32(const CUtensorMap& map, const Args& a, void* out, int* err, int model, int force,
                             bool walls, cudaStream_t s);
cudaError_t launch_fused_bf16(const CUtensorMap& map, const Args& a, void* out, int* err, int model, int force,
                              bool walls, cudaStream_t s);
cudaError_t launch_fused_f16(const CUtensorMap& map, const Args& a, void* out, int* err, int model, int force,
                             bool walls, cudaStream_t s);

// 2 or 4 steps of the unforced cascaded collision with round to nearest
// (lbm_multi.cuh) from a.f (natural layout, even step) into `out`; `map` describes a.f.
cudaError_t launch_multi_f32(const CUtensorMap& map, const Args& a, void* out, int* err, int steps, cudaStream_t s);
cudaError_t launch_multi_bf16(const CUtensorMap& map, const Args& a, void* out, int* err, int steps, cudaStream_t s);
cudaError_t launch_multi_f16(const CUtensorMap& map, const Args& a, void* out, int* err, int steps, cudaStream_t s);

// Steps t0 .. t0 + n - 1 of a small lattice in one launch (lbm_resident.cuh); n = 0
// only asks whether the device can run it.
cudaError_t launch_resident_f64(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s);
cudaError_t launch_resident_f32(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s);
cudaError_t launch_resident_bf16(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s);
cudaError_t launch_resident_f16(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s);

// Auxiliary kernels (lbm_aux.cu); every field argument is dense [..][ny][nx] FP64 device memory.
cudaError_t launch_init(const Args& a, int store, int model, int force, const double* rho, const double* u,
                        cudaStream_t s);
cudaError_t launch_set_f(const Args& a, int store, const double* f, cudaStream_t s);
cudaError_t launch_get_f(const Args& a, int store, bool odd, bool walls, double* f, cudaStream_t s);
cudaError_t launch_macros(const Args& a, int store, bool odd, bool walls, int force, double* rho, double* u,
                          cudaStream_t s);
cudaError_t launch_strain(const Args& a, int store, bool odd, bool walls, int force, double* out, cudaStream_t s);
// FP64 sums (rho, rho ux, rho uy) into partials[3 * nblocks] then out[3] (device).
int stats_blocks(const Args& a);
cudaError_t launch_stats(const Args& a, int store, bool odd, bool walls, int force, double* partials, double* out,
                         cudaStream_t s);

// Record the message returned by lbm_last_error() and return `code`.
int set_error(int code, const char* fmt, ...);

// dst[i] = (float)src[i], round to nearest.
cudaError_t launch_narrow(const double* src, float* dst, size_t n, cudaStream_t s);

}  // namespace lbm
