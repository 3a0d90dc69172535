// Fused lattice Boltzmann step: pull-stream + moving-wall bounce-back + moments + equilibrium +
// Knudsen sensor + per-tile sensor max + BGK collision, one pass over HBM.
//
// Paper (arXiv 1507.06767): streaming and collision of Sec. 2.2 (Eq. bgklb, collide-and-stream
// split), equilibrium Eq. (feq_i), moments Eqs. (rho), (u), sensor Eq. (sensor) / (kkn) of
// Sec. 3.2-3.3, moving bounce-back of Sec. 4.1.
//
// Thread mapping: a CTA of 32 x 8 threads covers 32 cells along x and 8 rows along y; in 3-D it
// walks 8 planes along z.  A CTA therefore owns whole 8^d base tiles (4 of them), so the tile maxima
// are written with plain stores: no atomics, no zeroing pass.  Each thread issues its q gathers
// before any arithmetic, so a warp keeps q independent coalesced loads in flight.
//
// Arithmetic is done on deviations from the rest state, df_i = f_i - w_i: rho - 1 = sum df_i and
// rho u = sum c_i df_i lose no digits to the large w_i, and f^neq = df_i - (f^eq_i - w_i) is formed
// without cancelling against w_i.
#pragma once

#include <atomic>

#include "lbm_internal.h"

namespace lbm {

constexpr int CTA_X = 32;
constexpr int CTA_Y = 8;
constexpr int TILE = 8;

// Tuning knobs (compile-time): resident CTAs per SM requested from the register allocator (one-cell
// kernel: 4 -> at most 64 registers, 1024 threads per SM; the two-cell kernel with 16-bit storage:
// 4, no spills, measured at 512^3 FP16 1.91 ms against 2.00 ms with 3; with FP32 storage: 3 -> at
// most 80 registers, no spills, 3.03 ms against 3.15 ms with 4), and cache hints of the population
// loads / stores (0: default, 1: read-only path / streaming store, 2: evict-first load, 3:
// read-only path asking L2 for the 256-byte group around each address: 512^3 FP16 two-cell 1.912
// -> 1.887 ms, FP32 one-cell 3.109 -> 3.074 ms, FP32 two-cell unchanged).  Measured on GB300 at
// 256^3 D3Q19 FP32: without a minimum the allocator takes 140 registers and the one-cell kernel
// runs at half speed.
#ifndef LBM_STEP_MIN_BLOCKS
#define LBM_STEP_MIN_BLOCKS 4
#endif
#ifndef LBM_PAIR_MIN_BLOCKS
#define LBM_PAIR_MIN_BLOCKS 4
#endif
#ifndef LBM_PAIR_MIN_BLOCKS_F32
#define LBM_PAIR_MIN_BLOCKS_F32 3
#endif
#ifndef LBM_LOAD_HINT
#define LBM_LOAD_HINT 3
#endif
#ifndef LBM_STORE_HINT
#define LBM_STORE_HINT 0
#endif
// 1: CTAs whose cells and all their pull sources lie inside the lattice take a gather without
// wall or wrap logic (one address offset per direction)
#ifndef LBM_INTERIOR_FAST
#define LBM_INTERIOR_FAST 1
#endif
// 1: rows inside in y and z but at an x face take gather_xsel (address selects, no branches)
#ifndef LBM_XSEL_PATH
#define LBM_XSEL_PATH 1
#endif

template <class T>
__device__ __forceinline__ T load_pop(const T *p) {
#if LBM_LOAD_HINT == 1 || LBM_LOAD_HINT == 3
    return __ldg(p);
#elif LBM_LOAD_HINT == 2
    return __ldcs(p);
#else
    return *p;
#endif
}

#if LBM_LOAD_HINT == 3
// read-only loads that also ask L2 to fetch the whole 256-byte sector group around the address
template <>
__device__ __forceinline__ float load_pop<float>(const float *p) {
    float v;
    asm("ld.global.nc.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
template <>
__device__ __forceinline__ float2 load_pop<float2>(const float2 *p) {
    float2 v;
    asm("ld.global.nc.L2::256B.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
template <>
__device__ __forceinline__ unsigned load_pop<unsigned>(const unsigned *p) {
    unsigned v;
    asm("ld.global.nc.L2::256B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
template <>
__device__ __forceinline__ unsigned short load_pop<unsigned short>(const unsigned short *p) {
    unsigned short v;
    asm("ld.global.nc.L2::256B.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
#endif

template <class T>
__device__ __forceinline__ void store_pop(T *p, T v) {
#if LBM_STORE_HINT == 1
    __stcs(p, v);
#else
    *p = v;
#endif
}

// Pull-gather of cell (x, y, z) in the general case (walls with moving-lid bounce-back, periodic
// wrap): writes the deviations from rest df_i = f_i - w_i of the populations arriving at the cell
// to df[i * STRIDE] (STRIDE 2 fills one lane of an array of pairs).  HALO: the faces of the slowest
// axis (z in 3-D, y in 2-D) may be cuts of a slab (StepParams::halo_lo / halo_hi); a source beyond
// such a face and inside the lattice along the other axes (or wrapped) is the neighbouring slab's
// cell, whose population i sits in the halo plane.  A source outside along another axis stays a
// wall ghost, and a 2-D slab whose high y face is a cut has no lid there.  The kernels without
// halos are instantiated with HALO = false and do not carry this code.
template <class L, int DT, int STRIDE = 1, bool HALO = false>
__device__ __forceinline__ void gather_cell(const typename Storage<DT>::T *__restrict__ fin,
                                            const StepParams &p, size_t N, int x, int y, int z,
                                            typename Storage<DT>::R *df) {
    using S = Storage<DT>;
    using R = typename S::R;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const bool perx = p.periodic & 1, pery = p.periodic & 2, perz = p.periodic & 4;
    // source coordinates x - c for c = +1 (xm) and c = -1 (xp), with their validity
    const int xm = (x == 0) ? nx - 1 : x - 1;
    const int xp = (x == nx - 1) ? 0 : x + 1;
    const bool vxm = (x > 0) || perx;
    const bool vxp = (x < nx - 1) || perx;
    const int ym = (y == 0) ? ny - 1 : y - 1;
    const int yp = (y == ny - 1) ? 0 : y + 1;
    const bool vym = (y > 0) || pery;
    const bool vyp = (y < ny - 1) || pery;  // false <=> the y+1 ghost is the lid
    int zm = z, zp = z;
    bool vzm = true, vzp = true;
    if (L::D == 3) {
        zm = (z == 0) ? nz - 1 : z - 1;
        zp = (z == nz - 1) ? 0 : z + 1;
        vzm = (z > 0) || perz;
        vzp = (z < nz - 1) || perz;
    }
    const int idx = (z * ny + y) * nx + x;
    const R lidx = param_lid_x<R>(p), lidz = param_lid_z<R>(p);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int cx = L::cx(i), cy = L::cy(i), cz = L::cz(i);
        const int sx = cx == 1 ? xm : (cx == -1 ? xp : x);
        const int sy = cy == 1 ? ym : (cy == -1 ? yp : y);
        const int sz = cz == 1 ? zm : (cz == -1 ? zp : z);
        const bool valid = (cx == 1 ? vxm : (cx == -1 ? vxp : true)) &&
                           (cy == 1 ? vym : (cy == -1 ? vyp : true)) &&
                           (cz == 1 ? vzm : (cz == -1 ? vzp : true));
        size_t src = valid ? (size_t)i * N + (size_t)((sz * ny + sy) * nx + sx)
                           : (size_t)L::opp(i) * N + (size_t)idx;
        const typename S::T *from = fin;
        bool lid = cy == -1 && !vyp;
        if constexpr (HALO) {
            const bool okx = cx == 1 ? vxm : (cx == -1 ? vxp : true);
            const bool oky = cy == 1 ? vym : (cy == -1 ? vyp : true);
            const bool okz = cz == 1 ? vzm : (cz == -1 ? vzp : true);
            const int cs = (L::D == 3) ? cz : cy;  // component along the slab axis
            const bool beyond = (L::D == 3) ? (cz != 0 && !okz && okx && oky)
                                            : (cy != 0 && !oky && okx);
            const void *hv = cs == 1 ? p.halo_lo : (cs == -1 ? p.halo_hi : nullptr);
            if (beyond && hv != nullptr) {
                from = static_cast<const typename S::T *>(hv);
                src = (L::D == 3) ? (size_t)i * ((size_t)nx * ny) + (size_t)(sy * nx + sx)
                                  : (size_t)i * nx + (size_t)sx;
            }
            if (L::D == 2 && p.halo_hi != nullptr) lid = false;
        }
        R v = S::to_r(load_pop(from + src));
        if (!S::SHIFTED) v -= weight<L, R>(i);  // w_opp(i) == w_i
        if (lid) {
            // moving lid: + 2 w_i (c_i . u_lid) / c_s^2, wall density 1
            v += R(6) * weight<L, R>(i) * (R(cx) * lidx + R(cz) * lidz);
        }
        df[i * STRIDE] = v;
    }
}

// Pull-gather of a cell whose q sources all lie inside the lattice (no wall, no wrap): population i
// comes from idx - (c_z plane + c_y nx + c_x) of population i's array.
template <class L, int DT>
__device__ __forceinline__ void gather_interior(const typename Storage<DT>::T *__restrict__ fin,
                                                size_t N, int nx, int plane, size_t idx,
                                                typename Storage<DT>::R *df) {
    using S = Storage<DT>;
    using R = typename S::R;
    const typename S::T *base = fin + idx;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const long long off =
            (long long)i * (long long)N - (long long)(L::cz(i) * plane + L::cy(i) * nx + L::cx(i));
        R v = S::to_r(load_pop(base + off));
        if (!S::SHIFTED) v -= weight<L, R>(i);
        df[i] = v;
    }
}

// Pull-gather of a cell whose y and z sources lie inside the lattice: as gather_interior, except
// that a pull along x that leaves the lattice (x = 0 pulling along +x, x = nx - 1 along -x)
// selects its address instead of branching: the wrapped cell on a periodic x axis, else the
// cell's own opposite population (bounce-back at a resting wall; the lid is a y wall).
template <class L, int DT>
__device__ __forceinline__ void gather_xsel(const typename Storage<DT>::T *__restrict__ fin,
                                            size_t N, int nx, int plane, size_t idx, int x,
                                            bool perx, typename Storage<DT>::R *df) {
    using S = Storage<DT>;
    using R = typename S::R;
    const typename S::T *base = fin + idx;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const int cx = L::cx(i);
        const long long off =
            (long long)i * (long long)N - (long long)(L::cz(i) * plane + L::cy(i) * nx + cx);
        const typename S::T *src = base + off;
        if (cx != 0) {
            const bool face = cx == 1 ? x == 0 : x == nx - 1;
            const typename S::T *alt = perx ? src + cx * nx : fin + (size_t)L::opp(i) * N + idx;
            src = face ? alt : src;
        }
        R v = S::to_r(load_pop(src));
        if (!S::SHIFTED) v -= weight<L, R>(i);
        df[i] = v;
    }
}

// Approximate FP32 reciprocal (PTX rcp.approx, max relative error about 1 ulp; inputs here are
// equilibrium populations, far from zero and from the subnormal range).
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Moments, equilibrium, sensor and BGK collision of one cell in FP32 from its gathered deviations df;
// emit(i, d) receives the post-collision deviation d = f*_i - w_i of every population.  Returns
// the sensor K (MODE != 0).
template <class L, int DT, int MODE, class Emit>
__device__ __forceinline__ typename Storage<DT>::R relax_cell(const typename Storage<DT>::R *df,
                                                              typename Storage<DT>::R omega,
                                                              Emit &&emit) {
    using S = Storage<DT>;
    using R = typename S::R;
    constexpr int Q = L::Q;
    // moments as deviations from rest
    R drho = 0, jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        drho += df[i];
        if (L::cx(i)) jx += R(L::cx(i)) * df[i];
        if (L::cy(i)) jy += R(L::cy(i)) * df[i];
        if (L::cz(i)) jz += R(L::cz(i)) * df[i];
    }
    const R rho = R(1) + drho;
    const R inv_rho = R(1) / rho;
    const R ux = jx * inv_rho, uy = jy * inv_rho, uz = jz * inv_rho;
    const R usq15 = R(1.5) * (ux * ux + uy * uy + uz * uz);

    R ksum = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const R cu = R(L::cx(i)) * ux + R(L::cy(i)) * uy + R(L::cz(i)) * uz;
        // P_i = c.u / cs2 + ((c.u)^2 - cs2 u.u) / (2 cs2^2)
        const R P = R(3) * cu + R(4.5) * cu * cu - usq15;
        const R w = weight<L, R>(i);
        const R dfeq = w * (drho + rho * P);  // f^eq_i - w_i
        const R fneq = df[i] - dfeq;
        if (MODE != 0) {
            // f^eq_i = (f^eq_i - w_i) + w_i: one add, one reciprocal, one fused multiply-add
            ksum = fmaf(fabsf(fneq), rcp_approx(dfeq + w), ksum);
        }
        emit(i, df[i] - omega * fneq);
    }
    return ksum * (R(1) / R(Q));
}

// relax_cell with the store of the post-collision populations at linear index idx.
template <class L, int DT, int MODE>
__device__ __forceinline__ typename Storage<DT>::R relax_store_cell(
    const typename Storage<DT>::R *df, typename Storage<DT>::R omega,
    typename Storage<DT>::T *__restrict__ fout, size_t N, int idx) {
    using S = Storage<DT>;
    using R = typename S::R;
    return relax_cell<L, DT, MODE>(df, omega, [&](int i, R dnew) {
        store_pop(fout + (size_t)i * N + idx,
                  S::from_r(S::SHIFTED ? dnew : dnew + weight<L, R>(i)));
    });
}

// Wait for the step before a 2-D step (launch_step_kernel).  The next one may start from here or, LATE,
// where the kernel says so at its end.
template <bool LATE, class T>
__device__ __forceinline__ T *step_wait(T *fin) {
    return LATE ? pdl_wait_only(fin) : pdl_wait(fin);
}

// The halo planes are read behind the wait too: the launch before the step may have filled them.
__device__ __forceinline__ void order_halos(StepParams &p) {
    p.halo_lo = pdl_order(p.halo_lo);
    p.halo_hi = pdl_order(p.halo_hi);
}

// The maxima of the warp's lanes of each tile (-1: none) into the tile's, one atomic a tile.
__device__ __forceinline__ void combine_tile_max(int tile, int kmax, float *tile_max) {
    const unsigned same = __match_any_sync(0xffffffffu, tile);
    const int m = __reduce_max_sync(same, kmax);
    if (tile >= 0 && (int)(threadIdx.x & 31) == __ffs(same) - 1)
        atomicMax(reinterpret_cast<int *>(tile_max) + tile, m);
}

// MODE 0: no sensor.  MODE 1: sensor and per-tile max.  MODE 2: MODE 1 plus per-cell K.  HALO:
// the faces of the slowest axis may be cuts of a slab (gather_cell).  FLAT (no halo): a CTA takes 256
// consecutive cells of a plane, wherever rows begin and end among them; CTAs share tiles then, whose
// maxima they combine with atomics in a buffer that the sensor step before has cleared.  LATE (2-D): see
// launch_step_kernel.
template <class L, int DT, int MODE, bool HALO = false, bool FLAT = false, bool LATE = false>
__global__ void __launch_bounds__(CTA_X *CTA_Y, LBM_STEP_MIN_BLOCKS)
    fused_step_kernel(const typename Storage<DT>::T *__restrict__ fin,
                      typename Storage<DT>::T *__restrict__ fout, StepParams p,
                      typename Storage<DT>::R *__restrict__ tile_max,
                      typename Storage<DT>::R *__restrict__ k_field) {
    using S = Storage<DT>;
    using R = typename S::R;
    using B = typename Bits<R>::type;
    constexpr int Q = L::Q;
    constexpr int ZT = (L::D == 3) ? TILE : 1;

    static_assert(!FLAT || !HALO, "flat rows have no halo");
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int lane = threadIdx.x;
    const int at = blockIdx.x * (CTA_X * CTA_Y) + threadIdx.y * CTA_X + lane;  // FLAT: in the plane
    const int y = FLAT ? at / nx : blockIdx.y * CTA_Y + threadIdx.y;
    const int x = FLAT ? at - y * nx : blockIdx.x * CTA_X + lane;
    const int z0 = blockIdx.z * ZT;
    const bool active = (x < nx) && (y < ny);
    const size_t N = (size_t)nx * ny * nz;
    const R omega = param_omega<R>(p);

    if constexpr (L::D == 2) fin = step_wait<LATE>(fin);
    if constexpr (L::D == 2 && HALO) order_halos(p);

    // clear the other tile buffer for the next sensor step (kernels that combine tiles across
    // CTAs with atomics need it zeroed)
    if (MODE != 0 && p.tile_zero) {
        const size_t nt = (size_t)p.ntx * p.nty * p.ntz;
        const size_t nthreads = (size_t)gridDim.x * gridDim.y * gridDim.z * blockDim.x * blockDim.y;
        const size_t me = (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                              (blockDim.x * blockDim.y) +
                          threadIdx.y * blockDim.x + threadIdx.x;
        for (size_t k = me; k < nt; k += nthreads) static_cast<R *>(p.tile_zero)[k] = R(0);
    }

    B kmax = 0;
    // a warp is one row of 32 cells: when the row and all its pull sources lie inside the lattice
    // (a warp-uniform test) the gather needs no wall or wrap logic.  FLAT: 32 cells of one row or more.
    bool inner_x = blockIdx.x * CTA_X >= 1 && (blockIdx.x + 1) * CTA_X <= nx - 1;
    bool inner_y = y >= 1 && y <= ny - 2;
    if constexpr (FLAT) {
        inner_x = __all_sync(0xffffffffu, !active || (x >= 1 && x <= nx - 2));
        inner_y = __all_sync(0xffffffffu, !active || inner_y);
    }

    for (int dz = 0; dz < ZT; ++dz) {
        const int z = z0 + dz;
        if (z >= nz) break;
        if (active) {
            const int idx = (z * ny + y) * nx + x;
            R df[Q];
            const bool inner_yz = inner_y && (L::D == 2 || (z >= 1 && z <= nz - 2));
            if (LBM_INTERIOR_FAST && inner_yz && inner_x)
                gather_interior<L, DT>(fin, N, nx, nx * ny, (size_t)idx, df);
            else if (LBM_XSEL_PATH && inner_yz)
                gather_xsel<L, DT>(fin, N, nx, nx * ny, (size_t)idx, x, p.periodic & 1, df);
            else
                gather_cell<L, DT, 1, HALO>(fin, p, N, x, y, z, df);
            const R K = relax_store_cell<L, DT, MODE>(df, omega, fout, N, idx);
            if (MODE != 0) {
                const B kb = max_bits(K);
                kmax = kb > kmax ? kb : kmax;
                if (MODE == 2) k_field[idx] = K;
            }
        }
    }

    if constexpr (LATE) pdl_start_next();
    if constexpr (FLAT && MODE != 0)
        combine_tile_max(active ? (blockIdx.z * p.nty + y / TILE) * p.ntx + x / TILE : -1, kmax,
                         tile_max);
    if (!FLAT && MODE != 0) {
        // max over the 8 lanes of each x-tile of this row, then over the 8 rows via shared memory
#pragma unroll
        for (int off = 4; off >= 1; off >>= 1) {
            const B o = __shfl_xor_sync(0xffffffffu, kmax, off);
            kmax = o > kmax ? o : kmax;
        }
        __shared__ B part[CTA_Y][CTA_X / TILE];
        if ((lane & (TILE - 1)) == 0) part[threadIdx.y][lane / TILE] = kmax;
        __syncthreads();
        if (threadIdx.y == 0 && lane < CTA_X / TILE) {
            B m = part[0][lane];
#pragma unroll
            for (int r = 1; r < CTA_Y; ++r) m = part[r][lane] > m ? part[r][lane] : m;
            const int tx = blockIdx.x * (CTA_X / TILE) + lane;
            if (tx < p.ntx) {
                const size_t t = ((size_t)blockIdx.z * p.nty + blockIdx.y) * p.ntx + tx;
                tile_max[t] = from_bits(m, R(0));
            }
        }
    }
}

// CTAs of a kernel that one SM and the GPU hold, asked for once.
struct Resident {
    int per_sm, all;
};
template <auto KERNEL>
inline Resident resident_ctas(int threads) {
    static std::atomic<int> known[CTA_Y + 1];  // by warps; 0: not asked yet
    static std::atomic<int> sms{0};
    const int warps = threads / CTA_X;
    int n = known[warps].load(std::memory_order_relaxed), m = sms.load(std::memory_order_relaxed);
    if (n == 0 || m == 0) {
        int dev = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, KERNEL, threads, 0) != cudaSuccess ||
            cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return {0, 0};
        known[warps].store(n, std::memory_order_relaxed);
        sms.store(m, std::memory_order_relaxed);
    }
    return {n, n * m};
}

// Launch of a step kernel.  In 2-D, where a step may take a few us, it overlaps its start with the
// end of the step before (launch_pdl): 128^2 FP64 4.62 -> 4.49 us a step in a graph, 6.16 -> 4.52 in calls
// of one step, 4096^2 FP32 170.9 either way.  In 3-D the CTAs that wait take the place of running ones:
// 195 x 129 x 97 FP32 78.0 -> 79.7 us, so not there.
//
// Waiting CTAs also settle where the step before has left room.  Where the GPU holds one step but not two, and
// one does not fill it, the next step's CTAs then lie unevenly over the SMs, up to the most an SM takes.
// So such a step (LATE) lets the next one start at the end of its CTAs: 320^2 FP64 27.6 -> 19.1 us (19.3 without
// overlap), with the sensor 45.5 -> 34.6 (36.9); 448^2 FP32 3.22 -> 2.83 (3.08), FP16 3.15 -> 2.70 (2.83).
// Elsewhere the early start gains: 128^2 FP64 4.61 -> 4.49, 480^2 FP32 3.47 -> 3.21, 900^2 FP16 6.07 ->
// 5.83.  Two kernels, as one that chooses at run time is scheduled around the choice: 1025 x 1023 FP16
// 9.77 -> 10.68.
template <class L, auto EARLY, auto LATE, class... Args>
inline cudaError_t launch_step_kernel(dim3 grid, dim3 block, cudaStream_t s, Args... args) {
    if constexpr (L::D == 3) {
        EARLY<<<grid, block, 0, s>>>(args...);
        return cudaGetLastError();
    } else {
        const Resident r = resident_ctas<EARLY>(block.x * block.y);
        const long long ctas = (long long)grid.x * grid.y;
        const bool late = r.per_sm > 0 && 2 * ctas > r.all && ctas <= r.all - r.all / r.per_sm;
        return launch_pdl(late ? LATE : EARLY, grid, block, 0, s, args...);
    }
}

template <class L, int DT, int MODE, bool HALO, bool FLAT, class... Args>
inline cudaError_t launch_step(dim3 grid, dim3 block, cudaStream_t s, Args... args) {
    return launch_step_kernel<L, fused_step_kernel<L, DT, MODE, HALO, FLAT>,
                              fused_step_kernel<L, DT, MODE, HALO, FLAT, L::D == 2>>(grid, block, s, args...);
}

// Whether a step takes the cells of a plane in a line (FLAT) rather than in rows of CTA_X lanes; dtype
// and the cells a lane takes along x as in the kernels.  Rows that do not fill whole warps leave lanes
// idle and start anywhere in a memory sector, a line neither (rows -> line, us a plain step: 195 x 129 x
// 97 FP32 76.3 -> 64.7, FP64 886 -> 773; 250 x 182 x 130 FP32 174 -> 144, BF16 101 -> 95; 100^3 FP16
// 29.7 -> 22.4; sensor steps of 100^3 FP32 39.2 -> 35.0, of 195 x 129 x 97 FP32 80.9 -> 69.0, FP16 67.4 ->
// 56.3, BF16 67.0 -> 55.9, of 251 x 181 x 131 FP16 128 -> 122).  Two cells a lane gain in long rows too, as
// a CTA then reads longer runs (256 x 256 x 128 FP16 124 -> 120, 128 x 128 x 64 unchanged); one cell a lane
// does not (256 x 256 x 64 FP32 101.0 -> 100.4), and two lose in sensor steps (250 x 182 x 130 BF16 102
// -> 105).  Below 2^19 cells the line has fewer than two CTAs an SM, where rows have more and smaller ones
// (42 x 36 x 227 FP32 18.7 -> 19.8 a sensor step, 40^3 9.8 -> 10.1), except in FP64, which the FP64 units
// bound (40^3 41 -> 29).  Over 47 lattices of odd sides above that line, FP32 and FP16 sensor steps gain
// 11 %; five of them lose 1 to 5 % in FP32 (151 x 191 x 25 25.1 -> 26.5, 166 x 59 x 99 31.8 -> 32.8), which
// neither the CTAs an SM nor the lanes saved tell apart from those that gain.  In 2-D FP64 (130^2 6.3 ->
// 4.9) and FP32 (50 x 700 2.10 -> 1.84, 301 x 203 2.22 -> 2.09) gain, 16-bit types lose (1025 x 1023 10.0 ->
// 10.5).
template <class L>
inline bool flat_rows(const StepParams &p, int mode, int dtype, int per_lane) {
    const long long plane = (long long)p.nx * p.ny;
    if (plane >= 1LL << 30) return false;  // the kernels count a plane's cells in ints
    const bool ragged = p.nx % (CTA_X * per_lane) != 0;
    if (dtype == 0) return mode == 0 && ragged;
    if (L::D == 2) return mode == 0 && ragged && dtype == 1 && per_lane == 1;
    if (plane * p.nz < 1LL << 19) return false;
    // a sensor step's tile maxima are combined in a buffer that has to be clear
    if (mode != 0) return ragged && per_lane == 1 && p.tile_clear;
    return ragged || (per_lane == 2 && p.nx >= 256);
}

template <class L, int DT, bool HALO = false>
cudaError_t launch_fused_step(const void *fin, void *fout, const StepParams &p, int mode,
                              void *tile_max, void *k_field, cudaStream_t stream) {
    using T = typename Storage<DT>::T;
    using R = typename Storage<DT>::R;
    const int zt = (L::D == 3) ? TILE : 1;
    dim3 block(CTA_X, CTA_Y, 1);
    dim3 grid((p.nx + CTA_X - 1) / CTA_X, (p.ny + CTA_Y - 1) / CTA_Y, (p.nz + zt - 1) / zt);
    const T *a = static_cast<const T *>(fin);
    T *b = static_cast<T *>(fout);
    R *tm = static_cast<R *>(tile_max);
    R *kf = static_cast<R *>(k_field);
    if constexpr (!HALO && (L::D == 3 || DT == 1)) {  // the types and modes that flat_rows takes
        if (flat_rows<L>(p, mode, DT, 1)) {
            grid.x = (unsigned)(((long long)p.nx * p.ny + CTA_X * CTA_Y - 1) / (CTA_X * CTA_Y));
            grid.y = 1;
            if constexpr (L::D == 3) {
                if (mode == 1)
                    return launch_step<L, DT, 1, false, true>(grid, block, stream, a, b, p, tm, kf);
                if (mode == 2)
                    return launch_step<L, DT, 2, false, true>(grid, block, stream, a, b, p, tm, kf);
            }
            return launch_step<L, DT, 0, false, true>(grid, block, stream, a, b, p, tm, kf);
        }
    }
    if (mode == 0)
        return launch_step<L, DT, 0, HALO, false>(grid, block, stream, a, b, p, tm, kf);
    if (mode == 1)
        return launch_step<L, DT, 1, HALO, false>(grid, block, stream, a, b, p, tm, kf);
    return launch_step<L, DT, 2, HALO, false>(grid, block, stream, a, b, p, tm, kf);
}

// A slab with halo faces (StepParams::halo_lo / halo_hi) runs the one-cell kernel with the halo
// gather; the other kernels do not take halos.
inline bool has_halo(const StepParams &p) { return p.halo_lo != nullptr || p.halo_hi != nullptr; }

}  // namespace lbm
