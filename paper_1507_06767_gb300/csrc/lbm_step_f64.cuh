// Fused step in FP64 (LBM_F64): the gathers of lbm_step.cuh, the relaxation of opposite directions in
// pairs.
#pragma once

#include "lbm_step.cuh"

namespace lbm {

// Constants of the relaxation, made once on the host.
struct RelaxF64 {
    double keep, half_keep;  // 1 - omega, (1 - omega) / 2
    double tau, neg_tau2;    // 1 / omega, -2 / omega
    double feq;              // omega / 36
    double kappa;            // 18 / omega
    double lam, lam_lo;      // omega / 12 in two parts: 12 lam is what a step leaves of the
                             // momentum's equilibrium, and one part's rounding would add up over
                             // the steps of a run
    explicit RelaxF64(const StepParams &p) {
        keep = 1.0 - p.omega;
        half_keep = 0.5 * keep;
        tau = 1.0 / p.omega;
        neg_tau2 = -2.0 * tau;
        feq = p.omega / 36.0;
        kappa = 18.0 * tau;
        lam = p.omega / 12.0;
        lam_lo = fma(-12.0, lam, p.omega) / 12.0;
    }
};

// Numerator and denominator of a sum of fractions |n_i| / e_i.
struct Fraction {
    double num, den;
};
__device__ __forceinline__ Fraction operator+(const Fraction &a, const Fraction &b) {
    return {fma(a.num, b.den, b.num * a.den), a.den * b.den};
}

// Whether |v| lies within 2^-300 .. 2^300, and whether v is finite, from the exponent.
__device__ __forceinline__ bool mid_range(double v) {
    return ((unsigned)__double2hiint(v) >> 20 & 0x7ff) - (1023 - 300) <= 600;
}
__device__ __forceinline__ bool is_finite(double v) {
    return ((unsigned)__double2hiint(v) >> 20 & 0x7ff) != 0x7ff;
}

// Moments, equilibrium, sensor and BGK collision of one cell from its gathered deviations df, as
// relax_cell; emit(i, d) receives the post-collision deviation of every population.
//
// FP64 runs at two multiply-adds per clock and SM here (1.25 TFLOP/s), so the step is bound by its
// count of FP64 instructions, not by memory.  Opposite directions are therefore relaxed together:
// with s = df_i + df_opp and m = df_i - df_opp,
//     f*_i - w, f*_opp - w = S +- M,   S = (1 - omega) / 2 s + omega w (B + 4.5 (c.j)^2 / rho),
//     M = (1 - omega) / 2 m + 3 omega w c.j,   B = rho - 1 - 1.5 j.j / rho,
// where j = rho u.  The momentum is scaled once by 3 omega w (w the diagonal weight), so that c.j is
// one addition in both S and M.  The sensor's fractions |f^neq| / f^eq are added over common
// denominators, three opposite pairs (two in 2-D) to one division.  mid (MODE != 0) comes back false
// where a pair's product of equilibria is so far from one that a product of three may leave the range
// (densities beyond 1e45, zeros, infinities, NaN) or a numerator overflows: the sensor is then
// sensor_cell_f64's.  That one gathers the cell again; kept at hand for it, the fractions took the 2-D
// kernel from 64 to 76 registers and a sensor step of 301 x 203 from 23.8 to 34.6 us.
//
// A plain D3Q19 step issues about 165 FP64 instructions a cell (about 350 with each direction relaxed
// by itself) and takes 0.653 ms at 128^3, 1.081 ms before, with the sensor 1.234 and 1.973; a D2Q9 step at
// 128^2 4.5 us, 10.9 us before (with the smaller CTAs below).  One warp alone waits for the longer chain of
// the sensor's sum (4000 x 1 with the sensor at every step 12.4 -> 14.3 us).  After 100 steps of a 128^2
// cavity the populations are 0.5e-16 to 1.3e-16 off an 80-bit evaluation, 2.2e-16 to 2.7e-16 before.
template <class L, int MODE, class Emit>
__device__ __forceinline__ double relax_cell_f64(const double *df, const RelaxF64 &k, bool &mid,
                                                 Emit &&emit) {
    constexpr int Q = L::Q;
    constexpr int GROUP = L::D == 3 ? 3 : 2;
    static_assert((Q - 1) / 2 % GROUP == 0, "whole groups of pairs");
    const double w0 = weight<L, double>(0);
    const double d0 = df[0];
    double s[Q], m[Q];  // entries i < opp(i)
    double drho = d0, j[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int o = L::opp(i);
        if (o < i) continue;
        s[i] = df[i] + df[o];
        m[i] = df[i] - df[o];
        drho += s[i];
        if (L::cx(i)) j[0] += double(L::cx(i)) * m[i];
        if (L::cy(i)) j[1] += double(L::cy(i)) * m[i];
        if (L::cz(i)) j[2] += double(L::cz(i)) * m[i];
    }
    // the scaled momentum j = 3 omega w rho u, w the diagonal weight, and v = kappa j with kappa =
    // 1 / (2 omega w rho): 4.5 omega w (c.j)^2 / rho is (c.j)(c.v) of these.  v is of the order of u, so no
    // product leaves the range where the populations do not.  The term in j.j takes the same factors,
    // so that the two cancel in the mass as far as they are rounded.
    const double inv_rho = 1.0 / (1.0 + drho);
    const double kappa = k.kappa * inv_rho;
    double jj = 0.0, v[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int d = 0; d < L::D; ++d) {
        j[d] = fma(j[d], k.lam, j[d] * k.lam_lo);
        v[d] = kappa * j[d];
        jj = fma(v[d], j[d], jj);
    }
    const double bd = fma(-1.0 / 3.0, jj, k.feq * drho);
    const double t0 = double(L::w36(0)) * bd;
    emit(0, fma(k.keep, d0, t0));
    double ksum = 0.0;  // twice the sum
    Fraction part = {0.0, 1.0};
    if (MODE != 0) {
        part = {fabs(fma(k.neg_tau2, t0, 2.0 * d0)), fma(k.tau, t0, w0)};
        mid = mid_range(part.den);
    }
    int held = 0;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        const int o = L::opp(i);
        if (o < i) continue;
        const double w = weight<L, double>(i);
        const double r = double(L::w36(i));  // the weight in diagonal weights: 1, axes 4 or 2
        double cj = 0.0, cv = 0.0;           // 3 omega w c.j
        bool first = true;
#pragma unroll
        for (int d = 0; d < L::D; ++d) {
            const int c = d == 0 ? L::cx(i) : d == 1 ? L::cy(i) : L::cz(i);
            if (!c) continue;
            cj = first ? double(c) * j[d] : cj + double(c) * j[d];
            cv = first ? double(c) * v[d] : cv + double(c) * v[d];
            first = false;
        }
        cj *= r;
        const double t = fma(cj, cv, r * bd);
        const double S = fma(k.half_keep, s[i], t), M = fma(k.half_keep, m[i], cj);
        emit(i, S + M);
        emit(o, S - M);
        if (MODE != 0) {
            // twice the non-equilibrium parts, and the equilibria
            const double ns = fma(k.neg_tau2, t, s[i]), nm = fma(k.neg_tau2, cj, m[i]);
            const double e = fma(k.tau, t, w), eo = k.tau * cj;
            const double np = ns + nm, nn = ns - nm, ep = e + eo, en = e - eo;
            const Fraction two = {fma(fabs(np), en, fabs(nn) * ep), ep * en};
            part = held == 0 && i != 1 ? two : part + two;
            mid = mid && mid_range(two.den);
            if (++held == GROUP) {
                mid = mid && is_finite(part.num);
                ksum += part.num / part.den;
                held = 0;
            }
        }
    }
    return ksum * (0.5 / double(Q));
}

// The sensor of one cell, each fraction divided by itself.
template <class L>
__device__ __forceinline__ double sensor_cell_f64(const double *df) {
    double drho = 0.0, u[3] = {0.0, 0.0, 0.0}, uu = 0.0, ksum = 0.0;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        drho += df[i];
        u[0] += double(L::cx(i)) * df[i];
        u[1] += double(L::cy(i)) * df[i];
        u[2] += double(L::cz(i)) * df[i];
    }
    const double rho = 1.0 + drho, inv_rho = 1.0 / rho;
    for (int d = 0; d < 3; ++d) {
        u[d] *= inv_rho;
        uu = fma(u[d], u[d], uu);
    }
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const double cu = double(L::cx(i)) * u[0] + double(L::cy(i)) * u[1] + double(L::cz(i)) * u[2];
        const double P = fma(4.5 * cu, cu, fma(3.0, cu, -1.5 * uu)), w = weight<L, double>(i);
        ksum += fabs(df[i] - w * fma(rho, P, drho)) / (w * rho * (1.0 + P));
    }
    return ksum * (1.0 / double(L::Q));
}

constexpr int F64_SPREAD_CTAS = 512;  // CTAs wanted of a plain step on a small 2-D lattice (152 SMs)

namespace f64 {  // by the name of the other types' one-cell kernel: a profile lists the FP64 step with them

// MODE, HALO, FLAT and LATE as in lbm::fused_step_kernel.  A CTA covers whole tiles as there where the step records
// the tile maxima; a plain step takes one plane a CTA in 3-D and, on small 2-D lattices, fewer rows
// (blockDim.y), as it is bound by the FP64 units: short CTAs shorten the last wave (128^3: 0.716 ms a
// step against 0.724 with two planes and 0.737 with four) and reach every SM (128^2: 512 CTAs of one
// row, 64 of eight).  The planes' CTAs come in a line, as there may be more than a grid's z takes.
template <class L, int MODE, bool HALO, bool FLAT = false, bool LATE = false>
__global__ void __launch_bounds__(CTA_X *CTA_Y, L::D == 3 ? 2 : MODE == 0 ? 5 : 4)
    fused_step_kernel(const double *__restrict__ fin, double *__restrict__ fout, StepParams p,
                      double *__restrict__ tile_max, double *__restrict__ k_field, const RelaxF64 k) {
    constexpr int Q = L::Q;
    constexpr int ZT = MODE != 0 && L::D == 3 ? TILE : 1;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int cta = CTA_X * blockDim.y;
    const int gx = FLAT ? (nx * ny + cta - 1) / cta : (nx + CTA_X - 1) / CTA_X;
    const int gy = FLAT ? 1 : (ny + blockDim.y - 1) / blockDim.y;
    const int bx = blockIdx.x % gx, by = blockIdx.x / gx % gy, bz = blockIdx.x / gx / gy;
    const int lane = threadIdx.x;
    const int at = bx * cta + threadIdx.y * CTA_X + lane;  // FLAT: in the plane
    const int y = FLAT ? at / nx : by * blockDim.y + threadIdx.y;
    const int x = FLAT ? at - y * nx : bx * CTA_X + lane, z0 = bz * ZT;
    const bool active = (x < nx) && (y < ny);
    const size_t N = (size_t)nx * ny * nz;
    if constexpr (L::D == 2) fin = step_wait<LATE>(fin);
    if constexpr (L::D == 2 && HALO) order_halos(p);
    if (MODE != 0 && p.tile_zero) {  // as in fused_step_kernel
        const size_t nt = (size_t)p.ntx * p.nty * p.ntz, me = (size_t)blockIdx.x * (CTA_X * CTA_Y) +
                                                              threadIdx.y * CTA_X + lane;
        for (size_t t = me; t < nt; t += (size_t)gridDim.x * (CTA_X * CTA_Y))
            static_cast<double *>(p.tile_zero)[t] = 0.0;
    }
    long long kmax = 0;
    bool inner_x = bx * CTA_X >= 1 && (bx + 1) * CTA_X <= nx - 1;
    bool inner_y = y >= 1 && y <= ny - 2;
    if constexpr (FLAT) {
        inner_x = __all_sync(0xffffffffu, !active || (x >= 1 && x <= nx - 2));
        inner_y = __all_sync(0xffffffffu, !active || inner_y);
    }
    for (int dz = 0; dz < ZT; ++dz) {
        const int z = z0 + dz;
        if (z >= nz) break;
        if (!active) continue;
        const int idx = (z * ny + y) * nx + x;
        double df[Q];
        const bool inner_yz = inner_y && (L::D == 2 || (z >= 1 && z <= nz - 2));
        if (inner_yz && inner_x)
            gather_interior<L, 0>(fin, N, nx, nx * ny, (size_t)idx, df);
        else if (inner_yz)
            gather_xsel<L, 0>(fin, N, nx, nx * ny, (size_t)idx, x, p.periodic & 1, df);
        else
            gather_cell<L, 0, 1, HALO>(fin, p, N, x, y, z, df);
        bool mid;
        double K = relax_cell_f64<L, MODE>(df, k, mid, [&](int i, double d) {
            fout[(size_t)i * N + idx] = d + weight<L, double>(i);
        });
        if (MODE != 0) {
            if (!mid) {
                gather_cell<L, 0, 1, HALO>(fin, p, N, x, y, z, df);
                K = sensor_cell_f64<L>(df);
            }
            const long long kb = max_bits(K);
            kmax = kb > kmax ? kb : kmax;
            if (MODE == 2) k_field[idx] = K;
        }
    }
    if constexpr (LATE) pdl_start_next();
    if (MODE != 0) {
        // max over the 8 lanes of each x-tile of this row, then over the 8 rows via shared memory
#pragma unroll
        for (int off = 4; off >= 1; off >>= 1) {
            const long long o = __shfl_xor_sync(0xffffffffu, kmax, off);
            kmax = o > kmax ? o : kmax;
        }
        __shared__ long long part[CTA_Y][CTA_X / TILE];
        if ((lane & (TILE - 1)) == 0) part[threadIdx.y][lane / TILE] = kmax;
        __syncthreads();
        if (threadIdx.y == 0 && lane < CTA_X / TILE) {
            long long m = part[0][lane];
#pragma unroll
            for (int r = 1; r < CTA_Y; ++r) m = part[r][lane] > m ? part[r][lane] : m;
            const int tx = bx * (CTA_X / TILE) + lane;
            if (tx < p.ntx)
                tile_max[((size_t)bz * p.nty + by) * p.ntx + tx] = from_bits(m, 0.0);
        }
    }
}

}  // namespace f64

template <class L, int MODE, bool HALO, bool FLAT, class... Args>
inline cudaError_t launch_step_f64(dim3 grid, dim3 block, cudaStream_t s, Args... args) {
    return launch_step_kernel<L, f64::fused_step_kernel<L, MODE, HALO, FLAT>,
                              f64::fused_step_kernel<L, MODE, HALO, FLAT, L::D == 2>>(grid, block, s, args...);
}

template <class L, bool HALO = false>
cudaError_t launch_fused_step_f64(const void *fin, void *fout, const StepParams &p, int mode,
                                  void *tile_max, void *k_field, cudaStream_t stream) {
    const int zt = mode != 0 && L::D == 3 ? TILE : 1;
    const long long gx = (p.nx + CTA_X - 1) / CTA_X, gz = (p.nz + zt - 1) / zt;
    int rows = CTA_Y;
    if (L::D == 2 && mode == 0)
        while (rows > 1 && gx * ((p.ny + rows - 1) / rows) < F64_SPREAD_CTAS) rows /= 2;
    const dim3 block(CTA_X, rows);
    dim3 grid((unsigned)(gx * ((p.ny + rows - 1) / rows) * gz));
    const double *a = static_cast<const double *>(fin);
    double *b = static_cast<double *>(fout), *tm = static_cast<double *>(tile_max),
           *kf = static_cast<double *>(k_field);
    const RelaxF64 k(p);
    if constexpr (!HALO) {
        if (mode == 0 && flat_rows<L>(p, mode, 0, 1)) {
            grid.x = (unsigned)(((long long)p.nx * p.ny + CTA_X * rows - 1) / (CTA_X * rows) * gz);
            return launch_step_f64<L, 0, false, true>(grid, block, stream, a, b, p, tm, kf, k);
        }
    }
    if (mode == 0)
        return launch_step_f64<L, 0, HALO, false>(grid, block, stream, a, b, p, tm, kf, k);
    if (mode == 1)
        return launch_step_f64<L, 1, HALO, false>(grid, block, stream, a, b, p, tm, kf, k);
    return launch_step_f64<L, 2, HALO, false>(grid, block, stream, a, b, p, tm, kf, k);
}

}  // namespace lbm
