// lbm_resident.cuh -- many time steps per launch for a small lattice that stays on
// chip (every storage kind, collision, force, edge and rounding).
//
// Up to about 100^2 nodes a step takes less than the gap between two launches (FP32
// 64^2: 1.3 us per step from a graph, of which the update is 0.3).  Here one cluster
// of up to 16 CTAs holds all populations in shared memory, a slab of rows per CTA
// and a node per thread, and takes every step of the call: the AA even step in the
// node's own slots, the odd step in the slots of its neighbours, which for the rows
// at a slab's edge lie in the shared memory of the next CTA (distributed shared
// memory; every slot still has one reader and writer).  A cluster barrier separates
// the steps; no CTA waits on memory.  The 18 slot addresses of a node are computed
// once and stay in registers.
//
// A step costs about 0.4 us of latency (barrier, loads, the collision's chain) plus
// instruction issue of five warps per SM quarter at most, so the lattice is spread
// over as many CTAs as a cluster takes (64^2 cavity: 0.87 us with 8, 0.69 with 16).
// Beyond one node per thread (800 a CTA, 80 registers each; fewer for the longer
// updates, resident_nodes) a launch per step over all 152 SMs wins: 128^2 1.8 us here
// with two rounds, 1.5 there.  An FP64 step costs its
// instructions (64 cycles each per warp and SM quarter), so beyond 128 nodes a CTA,
// one warp per quarter, the launch over all SMs wins; up to there what is saved is
// the launch and the filling of the chip.
// us per step, before -> now: FP32 periodic 16^2 1.2 -> 0.43, 64^2 1.3 -> 0.52, 101^2
// 1.35 -> 0.86; cavity 26^2 1.5 -> 0.64, 64^2 1.5 -> 0.69, 101^2 1.55 -> 1.02; raw-MRT forced
// cavity 101^2 1.6 -> 1.15; FP64 forced channel 4 x 32 5.87 -> 5.18, periodic 32^2 4.49 ->
// 3.77, cavity 32^2 5.35 -> 4.38, 128 x 16 5.22 -> 4.87 (128 nodes a CTA); in calls of 8 steps
// 4 x 32 5.96 -> 5.43, 128 x 16 5.37 -> 5.12.
#pragma once

#include "lbm_async.cuh"
#include "lbm_internal.h"

namespace lbm {

// Most threads of a CTA: 80 registers each; FP64 one warp per SM quarter (every further
// warp there costs as much as the first).
constexpr int resident_threads(int store) { return store == LBM_F64 ? 128 : 800; }
constexpr int kResidentMinSteps = 8;      // below, filling and emptying shared memory costs more than it saves
constexpr long kResidentMaxSteps = 16384; // of one launch (about 10 ms, FP64 100)

// CTAs of the cluster: a power of two, at most one per row.
inline int resident_size(const Args& a) {
    int size = 16;
    while (size > a.ny) size /= 2;
    return size;
}
// Most nodes of a CTA with which the steps on chip are no slower than a launch per step: a
// step costs its instructions on 16 SMs, so a force and stochastic rounding lower the
// line.  Speed of 512 steps on chip over 64-step graph replays, over the three
// collisions, periodic and cavity, with 16 or more rows (the lower end: slabs of one row):
//   FP32 stochastic, forced   480 nodes 0.96-1.36, 560 0.93-1.27, 707 0.88-1.05, 800 0.68-0.93
//   FP32 stochastic           640 1.04-1.31, 707 1.12-1.20, 784 0.94-1.11, 800 0.84-1.06
//   forced, FP32 and 16-bit   707 1.04-1.52, 784 0.94-1.25, 800 0.79-1.26
//   neither                   707 1.38-1.71, 784 1.26-1.54, 800 0.95-1.55
//   FP64                      128 0.99-1.3
// (112^2 FP32 stochastic with a force field: 2.15 us per step on chip, 1.67 launched.)
inline int resident_nodes(int store, int force, bool stochastic) {
    if (store == LBM_F64) return resident_threads(store);
    if (store == LBM_F32 && stochastic && force != 0) return 512;
    return force != 0 || stochastic ? 720 : resident_threads(store);
}
inline bool resident_fits(const Args& a, int store, int force) {
    const int size = resident_size(a);
    return (long long)((a.ny + size - 1) / size) * a.nx <= resident_nodes(store, force, a.rseed != 0);
}

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Address of this CTA's shared-memory location `addr` in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned cluster_addr(unsigned addr, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// Loads and stores through the cluster window (any CTA), and of this CTA's own
// shared memory by its plain address.
template <typename T> __device__ __forceinline__ T own_load(unsigned addr) {
    T v;
    if constexpr (sizeof(T) == 8) {
        unsigned long long w;
        asm volatile("ld.shared.b64 %0, [%1];" : "=l"(w) : "r"(addr) : "memory");
        __builtin_memcpy(&v, &w, 8);
    } else if constexpr (sizeof(T) == 4) {
        unsigned w;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(addr) : "memory");
        __builtin_memcpy(&v, &w, 4);
    } else {
        unsigned short w;
        asm volatile("ld.shared.b16 %0, [%1];" : "=h"(w) : "r"(addr) : "memory");
        __builtin_memcpy(&v, &w, 2);
    }
    return v;
}
template <typename T> __device__ __forceinline__ void own_store(unsigned addr, T v) {
    if constexpr (sizeof(T) == 8) {
        unsigned long long w;
        __builtin_memcpy(&w, &v, 8);
        asm volatile("st.shared.b64 [%0], %1;" ::"r"(addr), "l"(w) : "memory");
    } else if constexpr (sizeof(T) == 4) {
        unsigned w;
        __builtin_memcpy(&w, &v, 4);
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(w) : "memory");
    } else {
        unsigned short w;
        __builtin_memcpy(&w, &v, 2);
        asm volatile("st.shared.b16 [%0], %1;" ::"r"(addr), "h"(w) : "memory");
    }
}
template <typename T> __device__ __forceinline__ T cluster_load(unsigned addr) {
    T v;
    if constexpr (sizeof(T) == 8) {
        unsigned long long w;
        asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(w) : "r"(addr) : "memory");
        __builtin_memcpy(&v, &w, 8);
    } else if constexpr (sizeof(T) == 4) {
        unsigned w;
        asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(w) : "r"(addr) : "memory");
        __builtin_memcpy(&v, &w, 4);
    } else {
        unsigned short w;
        asm volatile("ld.shared::cluster.b16 %0, [%1];" : "=h"(w) : "r"(addr) : "memory");
        __builtin_memcpy(&v, &w, 2);
    }
    return v;
}
template <typename T> __device__ __forceinline__ void cluster_store(unsigned addr, T v) {
    if constexpr (sizeof(T) == 8) {
        unsigned long long w;
        __builtin_memcpy(&w, &v, 8);
        asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(addr), "l"(w) : "memory");
    } else if constexpr (sizeof(T) == 4) {
        unsigned w;
        __builtin_memcpy(&w, &v, 4);
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(addr), "r"(w) : "memory");
    } else {
        unsigned short w;
        __builtin_memcpy(&w, &v, 2);
        asm volatile("st.shared::cluster.b16 [%0], %1;" ::"r"(addr), "h"(w) : "memory");
    }
}

// One step of one node.  slot[p]: the address of the slot of plane p that the node
// reads and writes (own slots on even steps, through the cluster window for planes
// with e_p,y != 0 on odd ones); population q is read from slot[opp(q)] on odd steps,
// from slot[q] on even ones, and the results go back in AA order.  At a wall slot[opp(q)]
// is the node's own slot q for a link q that enters through the wall.
template <int MODEL, int STORE, int FORCE, bool SR, bool ODD>
__device__ __forceinline__ void resident_node(const Args& a, const Coef<typename Store<STORE>::R>& c, const unsigned slot[9],
                                              bool edge, int x, int y, unsigned rb) {
    using S = Store<STORE>;
    using T = typename S::T;
    using R = typename S::R;
    constexpr bool TS = SR && STORE == LBM_F32;
    R d[9], e[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const int p = ODD ? opp(q) : q;
        d[q] = S::dec(ODD && cy(p) != 0 ? cluster_load<T>(slot[p]) : own_load<T>(slot[p]));
    }
    if (ODD && edge) {
#pragma unroll
        for (int q = 1; q < 9; ++q) {
            const int w = incoming_wall(a, q, x, y);
            if (w >= 0) d[q] = add_wall_term<R>(a, d[q], q, w);
        }
    }
    R Fx, Fy;
    node_force<R, FORCE>(a, x, y, Fx, Fy);
    collide<MODEL, R, (FORCE != 0), TS>(d, Fx, Fy, c, e);
    if (ODD && edge) {
#pragma unroll
        for (int q = 1; q < 9; ++q) {
            const int w = incoming_wall(a, opp(q), x, y);
            if (w < 0) continue;
            if constexpr (TS) {
                float e2;
                d[q] = two_sum(d[q], wall_term<R>(a, opp(q), w), e2);
                e[q] = e[q] + e2;
            } else {
                d[q] = add_wall_term<R>(a, d[q], opp(q), w);
            }
        }
    }
    const unsigned rn = SR ? round_node(a, rb, x, y) : 0u;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const unsigned rw = rn + static_cast<unsigned>(q) * kRoundStride;
        T o;
        if constexpr (TS) o = round_sr32(d[q], e[q], rw);
        else if constexpr (SR) o = enc_sr<STORE>(d[q], rw);
        else o = S::enc(d[q]);
        const int p = ODD ? q : opp(q);
        if (ODD && cy(p) != 0) cluster_store<T>(slot[p], o);
        else own_store<T>(slot[p], o);
    }
}

// Steps t0 .. t0 + n - 1 of the whole lattice in place.  One cluster; CTA k holds
// ny / size rows (+ 1 for the first ny mod size CTAs), one thread per node.
template <int MODEL, int STORE, int FORCE, bool SR>
__global__ void __launch_bounds__(resident_threads(STORE), 1) resident_kernel(const Args a, unsigned long long t0, int n, int rows_max) {
    using T = typename Store<STORE>::T;
    using R = typename Store<STORE>::R;
    extern __shared__ __align__(16) unsigned char resident_smem[];
    T* A = reinterpret_cast<T*>(resident_smem);
    const unsigned k = cluster_rank(), size = cluster_size();
    const int q0 = a.ny / int(size), rem = a.ny - q0 * int(size);
    const int y0 = int(k) * q0 + min(int(k), rem), rows = q0 + (int(k) < rem ? 1 : 0);
    const int pl = rows_max * a.nx, i = threadIdx.x;
    const bool live = i < rows * a.nx;
    const int r = i / a.nx, x = i - r * a.nx, y = y0 + r;
    const bool edge = (x == 0 && a.wall[LBM_WEST]) || (x == a.nx - 1 && a.wall[LBM_EAST]) || (y == 0 && a.wall[LBM_SOUTH]) ||
                      (y == a.ny - 1 && a.wall[LBM_NORTH]);
    unsigned even[9], odd[9];
    {
        const unsigned plane = unsigned(pl) * sizeof(T), width = unsigned(a.nx) * sizeof(T), self = smem_addr(A);
        const unsigned kp = k > 0 ? k - 1 : size - 1, kn = k + 1 < size ? k + 1 : 0;
        const int rows_p = q0 + (int(kp) < rem ? 1 : 0);
        const unsigned row = self + unsigned(r) * width, rowc = cluster_addr(self, k) + unsigned(r) * width;
        const unsigned rowm = r > 0 ? rowc - width : cluster_addr(self, kp) + unsigned(rows_p - 1) * width;
        const unsigned rowp = r < rows - 1 ? rowc + width : cluster_addr(self, kn);
        const unsigned xc = unsigned(x) * sizeof(T), xm = (x > 0 ? xc : width) - unsigned(sizeof(T)),
                       xp = x < a.nx - 1 ? xc + unsigned(sizeof(T)) : 0u;
#pragma unroll
        for (int p = 0; p < 9; ++p) {
            even[p] = row + xc + unsigned(p) * plane;
            // plane p at x + e_p, or for a link q = opp(p) through a wall the node's own slot q
            if (incoming_wall(a, opp(p), x, y) >= 0) odd[p] = (cy(p) == 0 ? row : rowc) + xc + unsigned(opp(p)) * plane;
            else odd[p] = (cy(p) == 0 ? row : (cy(p) > 0 ? rowp : rowm)) + (cx(p) == 0 ? xc : (cx(p) > 0 ? xp : xm)) + unsigned(p) * plane;
        }
    }
    const Coef<R> c(a);
    T* f = static_cast<T*>(a.f) + (long long)y * a.pitch + x;
    pdl_wait();
    if (live) {
#pragma unroll
        for (int q = 0; q < 9; ++q) A[q * pl + i] = f[q * a.plane];
    }
    cluster_sync();
    for (int s = 0; s < n; ++s) {
        const unsigned long long t = t0 + s;
        if (live) {
            const unsigned rb = SR ? round_hash(a.rseed, t) : 0u;
            if (t & 1) resident_node<MODEL, STORE, FORCE, SR, true>(a, c, odd, edge, x, y, rb);
            else resident_node<MODEL, STORE, FORCE, SR, false>(a, c, even, false, x, y, rb);
        }
        cluster_sync();  // an odd step reads and writes the neighbours' slots
    }
    if (live) {
#pragma unroll
        for (int q = 0; q < 9; ++q) f[q * a.plane] = A[q * pl + i];
    }
}

// Launches the steps, or with n = 0 finds out whether the device can hold the cluster
// (cudaErrorNotSupported if not).
template <int MODEL, int STORE, int FORCE, bool SR>
static cudaError_t launch_resident_one(const Args& a, unsigned long long t0, int n, cudaStream_t s) {
    const int size = resident_size(a), rows_max = (a.ny + size - 1) / size;
    const size_t smem = size_t(9) * rows_max * a.nx * sizeof(typename Store<STORE>::T);
    // At most 28,800 bytes a CTA, so no shared memory has to be opted into.  A function's
    // attributes belong to all lattices and host threads: only ever set to one value.
    static_assert(size_t(9) * resident_threads(STORE) * sizeof(typename Store<STORE>::T) <= 48 * 1024, "no opt-in");
    auto kernel = resident_kernel<MODEL, STORE, FORCE, SR>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(size);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(unsigned(size));
    c.blockDim = dim3(unsigned(rows_max * a.nx + 31) / 32 * 32);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = at;
    if (n == 0) {
        c.numAttrs = 1;
        int clusters = 0;
        e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &c);
        return e != cudaSuccess ? e : (clusters > 0 ? cudaSuccess : cudaErrorNotSupported);
    }
    c.numAttrs = 2;
    return cudaLaunchKernelEx(&c, kernel, a, t0, n, rows_max);
}

template <int MODEL, int STORE, int FORCE>
static cudaError_t launch_resident_sr(const Args& a, unsigned long long t0, int n, cudaStream_t s) {
    if constexpr (STORE != LBM_F64) {
        if (a.rseed) return launch_resident_one<MODEL, STORE, FORCE, true>(a, t0, n, s);
    }
    return launch_resident_one<MODEL, STORE, FORCE, false>(a, t0, n, s);
}
template <int MODEL, int STORE>
static cudaError_t launch_resident_force(const Args& a, int force, unsigned long long t0, int n, cudaStream_t s) {
    switch (force) {
        case 0: return launch_resident_sr<MODEL, STORE, 0>(a, t0, n, s);
        case 1: return launch_resident_sr<MODEL, STORE, 1>(a, t0, n, s);
        default: return launch_resident_sr<MODEL, STORE, 2>(a, t0, n, s);
    }
}
template <int STORE>
static cudaError_t launch_resident_store(const Args& a, int model, int force, unsigned long long t0, int n, cudaStream_t s) {
    switch (model) {
        case LBM_CASCADED: return launch_resident_force<LBM_CASCADED, STORE>(a, force, t0, n, s);
        case LBM_BGK: return launch_resident_force<LBM_BGK, STORE>(a, force, t0, n, s);
        default: return launch_resident_force<LBM_RAWMRT, STORE>(a, force, t0, n, s);
    }
}

}  // namespace lbm
