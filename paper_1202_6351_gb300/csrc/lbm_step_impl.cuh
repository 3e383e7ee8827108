// lbm_step_impl.cuh -- the fused D2Q9 stream-and-collide kernel, instantiated
// once per storage type by lbm_step_<store>.cu.
//
// One thread per node (variant 0; variant 1 takes two rows per thread with
// packed FP32x2 arithmetic, variant 2 four nodes of a row per thread with
// 64-bit accesses for 16-bit stores): AA-pattern load of the nine populations
// with the wall links resolved (Eq. 24, Sec. III-A, III-C), decode of the
// stored deviations to FP32/FP64, macroscopic fields (Eq. 26-27), raw moments
// (Eq. 15), source (Eq. 13-14), cascaded kernel g3..g8 (Eq. 17-22) or a
// sibling collision, back-transform (Eq. 25), encode and AA-pattern store.
// All of it in registers, one launch per time step.
#pragma once

#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_vec.cuh"

namespace lbm {

// One node per thread.
//
// With walls, a warp that holds a node on the lattice edge takes the wall-aware
// path with all its lanes on odd steps: the lanes that need it and the others
// together cost one update, where a branch per node cost one of each, the whole
// latency of a launch on a small lattice (us per step: FP32 cavity 257^2 2.72 -> 2.08,
// 512^2 4.45 -> 3.55, FP64 channel 4 x 32 32.8 -> 17.3).
//
// LIN: nodes numbered row by row over the lanes instead of a row per warp, so
// a narrow or ragged lattice leaves no lanes idle.  FP64 updates are bound by
// the FP64 pipe, which takes 16 cycles per warp instruction and SM however many
// lanes are active: full warps, one per CTA so that they spread over all SMs (us per
// step: channel 4 x 32 17.3 -> 8.5, 101^2 9.9 -> 5.1, 257^2 27.5 -> 17.4).
template <int MODEL, int STORE, bool ODD, int FORCE, bool WALLS, bool SR = false, bool LIN = false>
__global__ void __launch_bounds__(kStepBX * kStepBY) step_kernel(const Args a) {
    int x, y;
    if (LIN) {
        const unsigned n = blockIdx.x * blockDim.x + threadIdx.x;
        y = int(n / unsigned(a.nx));
        x = int(n - unsigned(y) * unsigned(a.nx));
    } else {
        x = blockIdx.x * blockDim.x + threadIdx.x;
        y = blockIdx.y * blockDim.y + threadIdx.y;
    }
    const bool inside = x < a.nx && y < a.ny;
    const bool edge = WALLS && ODD &&
                      __any_sync(0xffffffffu, inside && ((x == 0) | (x == a.nx - 1) | (y == 0) | (y == a.ny - 1)));
    pdl_wait();
    if (!inside) return;
    const unsigned rb = SR ? round_base(a) : 0u;
    if (edge) step_node<MODEL, STORE, ODD, FORCE, WALLS && ODD, SR>(a, x, y, rb);
    else step_node<MODEL, STORE, ODD, FORCE, false, SR>(a, x, y, rb);
}

// One node per thread from a.f into a.fo (out of place; periodic lattices,
// FP32 and FP64 storage: the adjoint's forward and recomputed steps).
template <int MODEL, int STORE, bool ODD, int FORCE, bool SR>
__global__ void __launch_bounds__(kStepBX * kStepBY) step_kernel_oop(const Args a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    pdl_wait();
    if (x >= a.nx || y >= a.ny) return;
    step_node<MODEL, STORE, ODD, FORCE, false, SR, true>(a, x, y, SR ? round_base(a) : 0u);
}

// Two rows per thread (nodes (x, y) and (x, y + 1)) with packed FP32x2
// arithmetic; a pair that touches a wall edge takes the per-node wall path.
template <int MODEL, int STORE, bool ODD, int FORCE, bool WALLS>
__global__ void __launch_bounds__(kStepBX * kStepBY, 8) step_kernel_pair(const Args a) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = 2 * (blockIdx.y * blockDim.y + threadIdx.y);
    pdl_wait();
    if (x >= a.nx || y >= a.ny) return;
    const bool two = y + 1 < a.ny;
    if (WALLS && ((x == 0) | (x == a.nx - 1) | (y == 0) | (y + 1 >= a.ny - 1))) {
        step_node_split<MODEL, STORE, ODD, FORCE, true>(a, x, y);
        if (two) step_node_split<MODEL, STORE, ODD, FORCE, true>(a, x, y + 1);
        return;
    }
    step_pair<MODEL, STORE, ODD, FORCE>(a, x, y, two);
}

// N nodes of a row per thread (16-bit stores, no per-node force field);
// vectors that need a wrapped or wall neighbour take the per-node path.
// The CTA is bx x by threads with bx a multiple of 32, so the lanes of a warp
// hold consecutive vectors of one row (step_vec exchanges elements between
// neighbouring lanes on odd steps).
// Register budget per parity, as measured, in CTAs of 128 threads per SM
// (CTAs of 256 run 3-4 % slower).  Node pairs (the unforced cascaded collision):
// five on the even step, where six (80 registers) spill (98.5 against 102 us per
// FP16 4096^2 launch); on the odd step seven, six with stochastic rounding, which
// keeps two random words per pair (4096^2: 109.8 us per step with seven, 108.5
// with six, 115 with eight; cavity 8192^2 419, 431, 419).  Single nodes: the even
// step spills at 64 registers and gets 80 (six); the odd step runs faster with
// more warps at 64 (eight).
constexpr int kVecThreads = 128;
constexpr bool vec_pairs(int model, int force) { return model == LBM_CASCADED && force == 0; }
constexpr int vec_blocks(bool pairs, bool odd, bool sr) {
    return pairs ? (odd ? (sr ? 6 : 7) : 5) : (odd ? 8 : 6);
}

template <int N, int MODEL, int STORE, bool ODD, int FORCE, bool WALLS, bool SR>
__global__ void __launch_bounds__(kVecThreads, vec_blocks(vec_pairs(MODEL, FORCE), ODD, SR)) step_kernel_vec(const Args a) {
    const int x0 = N * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const bool inside = x0 < a.nx && y < a.ny;
    const bool vec = inside && (ODD ? (x0 >= N && x0 + N < a.nx && (!WALLS || (y > 0 && y < a.ny - 1)))
                                    : (x0 + N <= a.nx));
    const unsigned vmask = ODD ? __ballot_sync(0xffffffffu, vec) : 0u;
    pdl_wait();
    if (vec) {
        if constexpr (vec_pairs(MODEL, FORCE)) step_vec_pair<STORE, ODD, SR>(a, x0, y, vmask, threadIdx.x & 31);
        else step_vec<N, MODEL, STORE, ODD, FORCE, SR>(a, x0, y, vmask, threadIdx.x & 31);
    } else if (inside) {
        const int x1 = min(x0 + N, a.nx);
        const unsigned rb = SR ? round_base(a) : 0u;
        for (int x = x0; x < x1; ++x) step_node_split<MODEL, STORE, ODD, FORCE, WALLS, SR>(a, x, y, rb);
    }
}

// CTA of bx x (threads / bx) threads, bx halved (down to 32) while half of it
// still covers the `width` threads a row needs, so narrow lattices leave no
// threads idle.
static inline dim3 fit_block(int bx, int width, int threads = kStepBX * kStepBY) {
    if (bx % 32 != 0 || bx < 32 || bx > threads) bx = kStepBX < threads ? kStepBX : threads;  // lanes of a warp share a row
    while (bx > 32 && bx / 2 >= width) bx /= 2;
    return dim3(bx, threads / bx);
}

template <int N, int MODEL, int STORE, bool ODD, int FORCE, bool WALLS, bool SR>
static cudaError_t launch_vec(const Args& a, cudaStream_t s) {
    const int vecs = (a.nx + N - 1) / N;
    const dim3 block = fit_block(a.block_x > 0 ? a.block_x : kStepBX, vecs, kVecThreads);
    const dim3 grid((vecs + block.x - 1) / block.x, (a.ny + block.y - 1) / block.y);
    return launch_chain(step_kernel_vec<N, MODEL, STORE, ODD, FORCE, WALLS, SR>, grid, block, 0, s, a);
}

template <int MODEL, int STORE, bool ODD, int FORCE, bool WALLS>
static cudaError_t launch_one(const Args& a, cudaStream_t s) {
    if (a.fo) {  // out of place: periodic FP32 / FP64 only
        if constexpr ((STORE == LBM_F32 || STORE == LBM_F64) && !WALLS) {
            const dim3 block = fit_block(a.block_x > 0 ? a.block_x : kStepBX, a.nx);
            const dim3 grid((a.nx + block.x - 1) / block.x, (a.ny + block.y - 1) / block.y);
            if (a.rseed) return launch_chain(step_kernel_oop<MODEL, STORE, ODD, FORCE, true>, grid, block, 0, s, a);
            return launch_chain(step_kernel_oop<MODEL, STORE, ODD, FORCE, false>, grid, block, 0, s, a);
        }
        return cudaErrorNotSupported;
    }
    if constexpr (STORE == LBM_F32) {
        if (a.rseed) {  // stochastic rounding of FP32 stores: variant 0 only
            const dim3 block = fit_block(a.block_x > 0 ? a.block_x : kStepBX, a.nx);
            const dim3 grid((a.nx + block.x - 1) / block.x, (a.ny + block.y - 1) / block.y);
            return launch_chain(step_kernel<MODEL, STORE, ODD, FORCE, WALLS, true>, grid, block, 0, s, a);
        }
    }
    if constexpr (STORE == LBM_F16DEV || STORE == LBM_BF16DEV) {
        if (a.rseed) {  // stochastic rounding: variants 0 and 2 (variant 1 runs variant 0)
            if constexpr (FORCE != 2) {
                if (a.variant == 2) return launch_vec<4, MODEL, STORE, ODD, FORCE, WALLS, true>(a, s);
            }
            const dim3 block = fit_block(a.block_x > 0 ? a.block_x : kStepBX, a.nx);
            const dim3 grid((a.nx + block.x - 1) / block.x, (a.ny + block.y - 1) / block.y);
            return launch_chain(step_kernel<MODEL, STORE, ODD, FORCE, WALLS, true>, grid, block, 0, s, a);
        }
        if constexpr (FORCE != 2) {
            if (a.variant == 2) return launch_vec<4, MODEL, STORE, ODD, FORCE, WALLS, false>(a, s);
        }
    }
    if constexpr (STORE == LBM_F64) {  // one full warp per CTA
        const unsigned nodes = unsigned(a.nx) * unsigned(a.ny);
        return launch_chain(step_kernel<MODEL, STORE, ODD, FORCE, WALLS, false, true>, dim3((nodes + 31) / 32), dim3(32),
                            0, s, a);
    }
    const dim3 block = fit_block(a.block_x > 0 ? a.block_x : kStepBX, a.nx);
    const int bx = block.x, by = block.y;
    if constexpr (STORE != LBM_F64) {
        if (a.variant == 1) {
            const int rows = (a.ny + 1) / 2;
            const dim3 grid((a.nx + bx - 1) / bx, (rows + by - 1) / by);
            return launch_chain(step_kernel_pair<MODEL, STORE, ODD, FORCE, WALLS>, grid, block, 0, s, a);
        }
    }
    const dim3 grid((a.nx + bx - 1) / bx, (a.ny + by - 1) / by);
    return launch_chain(step_kernel<MODEL, STORE, ODD, FORCE, WALLS>, grid, block, 0, s, a);
}

template <int MODEL, int STORE, bool ODD, int FORCE>
static cudaError_t pick_walls(const Args& a, bool walls, cudaStream_t s) {
    return walls ? launch_one<MODEL, STORE, ODD, FORCE, true>(a, s) : launch_one<MODEL, STORE, ODD, FORCE, false>(a, s);
}

template <int MODEL, int STORE, bool ODD>
static cudaError_t pick_force(const Args& a, int force, bool walls, cudaStream_t s) {
    switch (force) {
        case 0: return pick_walls<MODEL, STORE, ODD, 0>(a, walls, s);
        case 1: return pick_walls<MODEL, STORE, ODD, 1>(a, walls, s);
        default: return pick_walls<MODEL, STORE, ODD, 2>(a, walls, s);
    }
}

template <int MODEL, int STORE>
static cudaError_t pick_parity(const Args& a, bool odd, int force, bool walls, cudaStream_t s) {
    return odd ? pick_force<MODEL, STORE, true>(a, force, walls, s) : pick_force<MODEL, STORE, false>(a, force, walls, s);
}

template <int STORE>
static cudaError_t launch_step_store(const Args& a, int model, bool odd, int force, bool walls, cudaStream_t s) {
    switch (model) {
        case LBM_CASCADED: return pick_parity<LBM_CASCADED, STORE>(a, odd, force, walls, s);
        case LBM_BGK: return pick_parity<LBM_BGK, STORE>(a, odd, force, walls, s);
        default: return pick_parity<LBM_RAWMRT, STORE>(a, odd, force, walls, s);
    }
}

}  // namespace lbm
