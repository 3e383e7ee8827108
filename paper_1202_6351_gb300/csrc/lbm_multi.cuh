// lbm_multi.cuh -- up to four time steps per launch (temporal blocking) for the
// unforced cascaded collision with round to nearest, FP32 and 16-bit storage:
// one read and one write of the populations per `steps` collide-and-stream
// steps (Eq. 23-24).  Variant 3 runs it where it applies and the two-step kernel
// (lbm_fused.cuh) otherwise.
//
// A CTA owns a TX x TY tile of nodes.  The tile's state at t + steps depends on
// the tile grown by `steps` nodes at t, which is brought into shared memory; the
// AA even and odd steps then alternate in place in that one buffer, each on the
// tile grown by the number of steps still to come (g): the even step on g nodes
// a side, the odd step on g - 1.  After an odd step the buffer holds the state in
// the natural layout.  Nodes of the grown regions are computed by several CTAs.
//
// What bounds it: the FP32 pipe.  A node pair costs 232 pipe cycles per warp
// (collide_cascaded_pair), 347 G collisions/s over the chip; HBM would allow 340
// G updates/s with four steps per transfer.  So the tile is as large as shared
// memory admits with two CTAs per SM (three with 16-bit storage) that overlap
// each other's loads and barriers, the halo's share of the collisions is kept
// small, and everything but the collision is kept off the issue slots:
//   - a thread takes two neighbouring nodes of a row, so an unshifted plane of a
//     pair is one 64-bit (16-bit storage: 32-bit) access.  Pairs of the even
//     step start at even columns and pairs of the odd step at odd ones, where six
//     of the nine planes, shifted by one column, are aligned again;
//   - TX + 2 H is 64: a warp takes a row of the region, one pair per lane, the
//     addresses of a row step differ by a constant, and no division or bank
//     conflict between row ends occurs (flat pair indices over 64 x 32 tiles: 22
//     conflicts per pair and warp instead of 10, 162.9 G against 170.9);
//   - nodes next to a wall are left out of the odd step's pairs and done one per
//     thread in a pass of their own on tiles that a wall touches.
// FP32 4096^2, G updates/s: 56 x 40 170.9, 56 x 24 (three CTAs per SM) 166.7, 64 x 32
// 163.1, 56 x 32 158.7, 64 x 16 150.4; two steps per launch 148.4 (64 x 16), 134
// (64 x 32); the two-step kernel 138.7.  FP16: 56 x 40 with three CTAs 175.9, two
// 163.8, 128 x 32 177.3; two-step kernel 135.9, four nodes per thread 152.8.
//
// Few such tiles do not fill the SMs, and a row of them with one ragged column puts the
// full ones on every other SM.  Then 32 x 16 tiles, loaded by every thread (most are edge
// tiles, which a tensor copy would have to patch).  us per step of 32 x 16 tiles | 56 x 40
// tiles | the two-step kernel: FP32 257^2 1.89 | 3.81 | 3.46, 384^2 2.47 | 3.59 | 3.45, 480^2
// 3.10 | 3.57, 512^2 4.13 | 3.56 | 4.56, 560^2 4.89 | 3.67, 600^2 5.10 | 5.28 | 5.53, 640^2
// 5.58 | 5.38, 700^2 6.37 | 5.76 | 6.60, 57 x 8000 6.42 | 9.01 | 7.34, 20 x 20000 6.64 | 11.77 |
// 13.2; FP16 480^2 3.17 | 3.57, 560^2 4.80 | 3.64, 600^2 5.00 | 5.29, 640^2 5.68 | 5.45.  Both go in
// waves of blocks (456 of the small; 152 alone on their SM, then 304 of the large), so
// multi_small_us and multi_large_us are what was measured, by number of tiles, and
// the smaller one wins.  One step per launch (variant 0) beats both below about 750^2:
// FP32 257^2 1.70, 384^2 2.18, 512^2 3.18, 600^2 3.92, 700^2 4.91.
//
// Up to two 56 x 40 tiles per SM (304) the third block that 16-bit storage has room for stays
// unused: 384 threads a block then, as for FP32 (FP16 640^2 5.47 -> 5.25, 560^2 3.64 ->
// 3.37, 1000 x 401 5.51 -> 5.34; the two-step kernel 5.33, 5.36, 5.33).
#pragma once

#include <cuda.h>

#include "lbm_async.cuh"
#include "lbm_internal.h"
#include "lbm_pair.cuh"
#include "lbm_vec.cuh"

namespace lbm {

constexpr int kMultiSteps = 4;  // halo of the shared-memory box, the most steps of a launch

template <int STORE_, int TX_, int TY_, int NT_, int MINB_, bool TMA_>
struct MultiGeom {
    static constexpr int STORE = STORE_, TX = TX_, TY = TY_, H = kMultiSteps, NT = NT_, MINB = MINB_;
    static constexpr bool TMA = TMA_;
    static constexpr bool ROW = TX / 2 + H == 32;  // a warp takes a row of pairs, else pairs are numbered flat
    using T = typename Store<STORE>::T;
    static constexpr int ALIGN = 16 / int(sizeof(T));
    static constexpr int HX = (H + ALIGN - 1) / ALIGN * ALIGN;  // halo columns, 16-byte aligned for TMA
    static constexpr int BW = TX + 2 * HX, BH = TY + 2 * H;
    static constexpr int PLANE = BW * BH;
    static constexpr size_t SMEM = size_t(9) * PLANE * sizeof(T);
    static_assert(TX % 2 == 0 && (TX * sizeof(T)) % 16 == 0 && (BW * sizeof(T)) % 16 == 0, "aligned rows");
    static_assert(BW <= 256 && BH <= 256, "TMA box");
};
template <int STORE> struct MultiLarge : MultiGeom<STORE, 56, 40, 256, 3, true> {};
template <> struct MultiLarge<LBM_F32> : MultiGeom<LBM_F32, 56, 40, 384, 2, true> {};
template <int STORE> struct MultiWide : MultiGeom<STORE, 56, 40, 384, 2, true> {};
template <int STORE> struct MultiSmall : MultiGeom<STORE, 32, 16, 256, 3, false> {};

enum : int { kMultiErrTimeout = 1 };

// Two neighbouring nodes of a plane in shared memory (p aligned to the pair).
template <int STORE> struct PairIO {
    using T = typename Store<STORE>::T;
    static __device__ __forceinline__ float2 ld2(const T* p) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
        return make_float2(Half16<STORE>::lo(w), Half16<STORE>::hi(w));
    }
    static __device__ __forceinline__ void st2(T* p, float2 v) {
        *reinterpret_cast<uint32_t*>(p) = Half16<STORE>::pack(v.x, v.y);
    }
};
template <> struct PairIO<LBM_F32> {
    static __device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
    static __device__ __forceinline__ void st2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
};

// The pairs of a region of `rows` rows and `pw` pairs a row, box row and column
// (row0, col0) first: fn(pair's address, box row, box column) for each pair of this thread.
template <class G, typename Fn>
__device__ __forceinline__ void multi_pairs(typename G::T* A, int row0, int col0, int rows, int pw, Fn&& fn) {
    if constexpr (G::ROW) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (lane >= pw) return;
        typename G::T* p = A + (row0 + warp) * G::BW + col0 + 2 * lane;
        for (int r = warp; r < rows; r += G::NT / 32, p += (G::NT / 32) * G::BW) fn(p, row0 + r, col0 + 2 * lane);
    } else {
        const int n = pw * rows, dr = G::NT / pw, dc = G::NT - dr * pw;
        int r = int((threadIdx.x + 0.5f) * __frcp_rn(float(pw)));  // exact: threadIdx.x < 2^10
        int c = threadIdx.x - r * pw;
        for (int i = threadIdx.x; i < n; i += G::NT) {
            fn(A + (row0 + r) * G::BW + col0 + 2 * c, row0 + r, col0 + 2 * c);
            r += dr;
            c += dc;
            if (c >= pw) { c -= pw; ++r; }
        }
    }
}

// AA even step: every node of the region collides in its own slots.
template <class G>
__device__ __forceinline__ void multi_even(typename G::T* A, int g, int tw, int th, const float* __restrict__ kc) {
    using IO = PairIO<G::STORE>;
    multi_pairs<G>(A, G::H - g, G::HX - g, th + 2 * g, tw / 2 + g, [&](typename G::T* p, int, int) {
        float2 d[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) d[q] = IO::ld2(p + q * G::PLANE);
        collide_cascaded_pair(d, kc);
#pragma unroll
        for (int q = 0; q < 9; ++q) IO::st2(p + opp(q) * G::PLANE, d[q]);
    });
}

// AA odd step: population q arrives from slot opp(q) of the node at x - e_q and
// leaves into slot q of the node at x + e_q; each slot is read and written by one
// node only.  WL: nodes outside box columns xlo .. xhi or rows ylo .. yhi (next
// to a wall, or beyond it) are left alone.
template <class G, bool WL>
__device__ __forceinline__ void multi_odd(typename G::T* A, int g, int tw, int th, const float* __restrict__ kc, int xlo,
                                          int xhi, int ylo, int yhi) {
    using IO = PairIO<G::STORE>;
    using S = Store<G::STORE>;
    using T = typename G::T;
    multi_pairs<G>(A, G::H - g, G::HX - g, th + 2 * g, tw / 2 + g, [&](T* p, int row, int col) {
        bool m0 = true, m1 = true;
        if (WL) {
            const bool in = row >= ylo && row <= yhi;
            m0 = in && col >= xlo && col <= xhi;
            m1 = in && col + 1 >= xlo && col + 1 <= xhi;
            if (!m0 && !m1) return;
        }
        float2 d[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const T* s = p + opp(q) * G::PLANE - cy(q) * G::BW - cx(q);
            if (cx(q) != 0) d[q] = IO::ld2(s);
            else d[q] = make_float2(S::dec(s[0]), S::dec(s[1]));
        }
        collide_cascaded_pair(d, kc);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            T* s = p + q * G::PLANE + cy(q) * G::BW + cx(q);
            if (cx(q) != 0 && (!WL || (m0 && m1))) {
                IO::st2(s, d[q]);
            } else {
                if (!WL || m0) s[0] = S::enc(d[q].x);
                if (!WL || m1) s[1] = S::enc(d[q].y);
            }
        }
    });
}

// The odd step of the nodes next to a wall, one per thread: the south and north
// rows of the region, then the west and east columns between them.
template <class G>
__device__ __forceinline__ void multi_wall_nodes(const Args& a, typename G::T* A, int g, int x0, int y0) {
    using S = Store<G::STORE>;
    using T = typename G::T;
    const Coef<float> c(a);
    const bool wx = a.wall[LBM_WEST], wy = a.wall[LBM_SOUTH];
    const int X0 = wx ? max(x0 - g, 0) : x0 - g, X1 = wx ? min(x0 + G::TX + g, a.nx) : x0 + G::TX + g;
    const int Y0 = wy ? max(y0 - g, 0) : y0 - g, Y1 = wy ? min(y0 + G::TY + g, a.ny) : y0 + G::TY + g;
    const int w = X1 - X0;
    const bool south = wy && Y0 == 0, north = wy && Y1 == a.ny, west = wx && X0 == 0, east = wx && X1 == a.nx;
    const int ya = Y0 + (south ? 1 : 0), h = Y1 - (north ? 1 : 0) - ya;
    const int c0 = south ? w : 0, c1 = c0 + (north ? w : 0), c2 = c1 + (west ? h : 0), c3 = c2 + (east ? h : 0);
    for (int i = threadIdx.x; i < c3; i += G::NT) {
        int gx, gy;
        if (i < c0) { gx = X0 + i; gy = 0; }
        else if (i < c1) { gx = X0 + (i - c0); gy = a.ny - 1; }
        else if (i < c2) { gx = 0; gy = ya + (i - c1); }
        else { gx = a.nx - 1; gy = ya + (i - c2); }
        T* p = A + (gy - y0 + G::H) * G::BW + (gx - x0 + G::HX);
        float d[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int wl = incoming_wall(a, q, gx, gy);
            if (wl >= 0) d[q] = add_wall_term<float>(a, S::dec(p[q * G::PLANE]), q, wl);
            else d[q] = S::dec(p[opp(q) * G::PLANE - cy(q) * G::BW - cx(q)]);
        }
        collide_cascaded<float, false>(d, 0.f, 0.f, c);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const int wl = incoming_wall(a, opp(q), gx, gy);
            if (wl >= 0) p[opp(q) * G::PLANE] = S::enc(add_wall_term<float>(a, d[q], opp(q), wl));
            else p[q * G::PLANE + cy(q) * G::BW + cx(q)] = S::enc(d[q]);
        }
    }
}

__device__ __forceinline__ int wrap_mod(int v, int n) {
    if (v >= 0 && v < n) return v;
    v %= n;
    return v < 0 ? v + n : v;
}

// Fetches the box cell of lattice node (gx, gy) (a periodic image where it lies
// outside) with plain loads.
template <class G>
__device__ __forceinline__ void multi_fetch(const Args& a, const typename G::T* __restrict__ f, typename G::T* A, int x0,
                                            int y0, int gx, int gy) {
    using T = typename G::T;
    T* p = A + (gy - y0 + G::H) * G::BW + (gx - x0 + G::HX);
    const T* src = f + ((long long)wrap_mod(gy, a.ny) * a.pitch + wrap_mod(gx, a.nx));
#pragma unroll
    for (int q = 0; q < 9; ++q) p[q * G::PLANE] = src[q * a.plane];
}

// The region of the tile at (x0, y0) by one TMA load, which leaves zeros beyond the
// lattice; across a periodic edge the cells within `steps` nodes of the lattice are
// then fetched from their images (rows first, then columns between them).  Region
// cells further out, and cells beyond a wall, feed no node of the tile.  Returns
// false if the load did not land within a second (err is set).
template <class G>
__device__ __forceinline__ bool multi_load_tma(const CUtensorMap* map, const Args& a, const typename G::T* __restrict__ f,
                                               typename G::T* A, int* err, int x0, int y0, int steps,
                                               unsigned long long* bar, int* ok) {
    const int tid = threadIdx.x;
    const bool perx = !a.wall[LBM_WEST], pery = !a.wall[LBM_SOUTH];
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, static_cast<unsigned>(G::SMEM));
        tma_load_3d(A, map, x0 - G::HX, y0 - G::H, 0, bar);
        const bool done = mbar_wait_bounded(bar, 0, 1000000000ull);
        if (!done) {
            atomicOr(err, kMultiErrTimeout);
            mbar_wait_bounded(bar, 0, 4000000000ull);  // let the copy land before the CTA exits
        }
        *ok = done ? 1 : 0;
    }
    __syncthreads();
    if (!*ok) return false;
    if ((perx && (x0 - steps < 0 || x0 + G::TX + steps > a.nx)) || (pery && (y0 - steps < 0 || y0 + G::TY + steps > a.ny))) {
        const int X0 = x0 - steps, X1 = min(x0 + G::TX + steps, a.nx + steps);
        const int Y0 = y0 - steps, Y1 = min(y0 + G::TY + steps, a.ny + steps);
        const int xi0 = max(X0, 0), xi1 = min(X1, a.nx), yi0 = max(Y0, 0), yi1 = min(Y1, a.ny);
        const int rlo = pery ? max(0, min(0, Y1) - Y0) : 0, rhi = pery ? max(0, Y1 - max(a.ny, Y0)) : 0;
        const int rx0 = perx ? X0 : xi0, rw = max(0, (perx ? X1 : xi1) - rx0);
        const int clo = perx ? max(0, min(0, X1) - X0) : 0, chi = perx ? max(0, X1 - max(a.nx, X0)) : 0;
        const int ch = max(0, yi1 - yi0);
        const int nrow = (rlo + rhi) * rw, ncell = nrow + (clo + chi) * ch;
        for (int k = tid; k < ncell; k += G::NT) {
            int gx, gy;
            if (k < nrow) {
                const int r = k / rw;
                gx = rx0 + (k - r * rw);
                gy = r < rlo ? Y0 + r : max(a.ny, Y0) + (r - rlo);
            } else {
                const int c = (k - nrow) / ch;
                gy = yi0 + (k - nrow - c * ch);
                gx = c < clo ? X0 + c : max(a.nx, X0) + (c - clo);
            }
            multi_fetch<G>(a, f, A, x0, y0, gx, gy);
        }
        __syncthreads();
    }
    return true;
}

// The same region cell by cell, every thread its share (32-bit cells by
// asynchronous copies, all in flight at once).
template <class G>
__device__ __forceinline__ void multi_load_cells(const Args& a, const typename G::T* __restrict__ f, typename G::T* A,
                                                 int x0, int y0, int steps) {
    using T = typename G::T;
    const bool perx = !a.wall[LBM_WEST], pery = !a.wall[LBM_SOUTH];
    const int W = G::TX + 2 * steps, n = W * (G::TY + 2 * steps);
    for (int i = threadIdx.x; i < n; i += G::NT) {
        const int r = i / W, gx = x0 - steps + (i - r * W), gy = y0 - steps + r;
        if ((!perx && (gx < 0 || gx >= a.nx)) || (!pery && (gy < 0 || gy >= a.ny))) continue;
        if constexpr (sizeof(T) == 4) {
            const unsigned p = smem_addr(A + (gy - y0 + G::H) * G::BW + (gx - x0 + G::HX));
            const T* src = f + ((long long)wrap_mod(gy, a.ny) * a.pitch + wrap_mod(gx, a.nx));
#pragma unroll
            for (int q = 0; q < 9; ++q)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(p + unsigned(q * G::PLANE * sizeof(T))),
                             "l"(src + q * a.plane) : "memory");
        } else {
            multi_fetch<G>(a, f, A, x0, y0, gx, gy);
        }
    }
    if constexpr (sizeof(T) == 4) asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
}

// `steps` (2 or 4) steps of one tile from `in` (natural layout, even step) into `out`.
// smem holds G::SMEM bytes (1024-byte aligned); bar and ok live in shared memory
// and serve this tile only.  Every thread of the CTA calls this alike.
template <class G>
__device__ __forceinline__ void multi_tile(const CUtensorMap* map, const Args& a, const void* in, void* out, int* err, int x0,
                                           int y0, int steps, unsigned char* smem, unsigned long long* bar, int* ok) {
    using T = typename G::T;
    T* A = reinterpret_cast<T*>(smem);
    const int tid = threadIdx.x;
    const bool perx = !a.wall[LBM_WEST], pery = !a.wall[LBM_SOUTH];
    const T* f = static_cast<const T*>(in);
    if constexpr (G::TMA) {
        if (!multi_load_tma<G>(map, a, f, A, err, x0, y0, steps, bar, ok)) return;
    } else {
        multi_load_cells<G>(a, f, A, x0, y0, steps);
    }
    // the part of the tile inside the lattice (columns rounded up to whole pairs)
    const int tw = min(G::TX, (a.nx - x0 + 1) & ~1), th = min(G::TY, a.ny - y0);
    const bool near_wall = (!perx && (x0 - steps < 1 || x0 + G::TX + steps > a.nx - 1)) ||
                           (!pery && (y0 - steps < 1 || y0 + G::TY + steps > a.ny - 1));
    // box columns and rows of the nodes not next to a wall
    const int xlo = perx ? 0 : 1 - x0 + G::HX, xhi = perx ? G::BW : a.nx - 2 - x0 + G::HX;
    const int ylo = pery ? 0 : 1 - y0 + G::H, yhi = pery ? G::BH : a.ny - 2 - y0 + G::H;
#pragma unroll 1
    for (int g = steps; g > 0; g -= 2) {
        multi_even<G>(A, g, tw, th, a.kf);
        __syncthreads();
        if (near_wall) {
            multi_odd<G, true>(A, g - 1, tw, th, a.kf, xlo, xhi, ylo, yhi);
            multi_wall_nodes<G>(a, A, g - 1, x0, y0);
        } else {
            multi_odd<G, false>(A, g - 1, tw, th, a.kf, xlo, xhi, ylo, yhi);
        }
        if (g == 2) fence_async_shared();  // the last writes before the bulk stores read them
        __syncthreads();
    }
    T* fo = static_cast<T*>(out);
    if (x0 + G::TX <= a.nx) {  // one bulk copy per row and plane
        for (int j = tid; j < 9 * th; j += G::NT) {
            const int q = j / th, ty = j - q * th;
            bulk_store(fo + q * a.plane + (long long)(y0 + ty) * a.pitch + x0, A + q * G::PLANE + (ty + G::H) * G::BW + G::HX,
                       unsigned(G::TX * sizeof(T)));
        }
        bulk_commit();
        bulk_wait_read<0>();  // shared memory stays allocated until the copies have read it
    } else {
        const int w = a.nx - x0;
        for (int k = tid; k < w * th; k += G::NT) {
            const int ty = k / w, tx = k - ty * w;
            const T* p = A + (ty + G::H) * G::BW + (tx + G::HX);
            T* dst = fo + ((long long)(y0 + ty) * a.pitch + (x0 + tx));
#pragma unroll
            for (int q = 0; q < 9; ++q) dst[q * a.plane] = p[q * G::PLANE];
        }
    }
}

template <class G>
__global__ void __launch_bounds__(G::NT, G::MINB)
    multi_kernel(const __grid_constant__ CUtensorMap map, const Args a, const void* in, void* out, int* err, int steps) {
    extern __shared__ __align__(1024) unsigned char multi_smem[];
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int ok;
    pdl_wait();
    multi_tile<G>(&map, a, in, out, err, blockIdx.x * G::TX, blockIdx.y * G::TY, steps, multi_smem, &bar, &ok);
}

template <class G>
static cudaError_t launch_multi_geom(const CUtensorMap& map, const Args& a, void* out, int* err, int steps, cudaStream_t s) {
    const cudaError_t e =
        cudaFuncSetAttribute(multi_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(G::SMEM));
    if (e != cudaSuccess) return e;
    return launch_chain(multi_kernel<G>, dim3((a.nx + G::TX - 1) / G::TX, (a.ny + G::TY - 1) / G::TY), dim3(G::NT), G::SMEM,
                        s, map, a, static_cast<const void*>(a.f), out, err, steps);
}

// us per step of n tiles of 32 x 16 and of n full tiles of 56 x 40 nodes, FP32, as measured
// (above); a lattice without walls has more halo to patch.
inline double multi_small_us(double n) {
    return n <= 152 ? 1.9 : n <= 304 ? 2.5 : n <= 456 ? 3.1 : n <= 554 ? 4.1 : 1.0 + 0.0056 * n;
}
inline double multi_large_us(double n, bool walls) {
    return n <= 152 ? 3.6 : n <= 304 ? (walls ? 5.2 : 5.4) : 2.4 + 0.0132 * n;
}

template <int STORE>
static cudaError_t launch_multi_store(const CUtensorMap& map, const Args& a, void* out, int* err, int steps,
                                      cudaStream_t s) {
    using Large = MultiLarge<STORE>;
    using Small = MultiSmall<STORE>;
    const int gx = (a.nx + Large::TX - 1) / Large::TX, gy = (a.ny + Large::TY - 1) / Large::TY;
    const double full = gx * (a.ny + 5.0 * gy) / (Large::TY + 5);  // a tile costs its rows plus five, whatever its width
    const double small = double((a.nx + Small::TX - 1) / Small::TX) * ((a.ny + Small::TY - 1) / Small::TY);
    if (multi_small_us(small) < multi_large_us(full, a.wall[LBM_WEST] || a.wall[LBM_SOUTH]))
        return launch_multi_geom<Small>(map, a, out, err, steps, s);
    if constexpr (STORE != LBM_F32) {
        if ((long long)gx * gy <= 304) return launch_multi_geom<MultiWide<STORE>>(map, a, out, err, steps, s);
    }
    return launch_multi_geom<Large>(map, a, out, err, steps, s);
}

}  // namespace lbm
