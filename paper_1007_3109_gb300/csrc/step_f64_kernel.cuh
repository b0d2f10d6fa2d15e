// FP64 per-site update, shared by the single-simulation and batched kernels.
//
// One site: pull f_i(x, t + 1) = f*_i(x - e_i, t) (periodic), rho_s = sum_i f_i
// in index order, R_s(rho) from the reaction, then Eq. relax
//   post = f + (w_i rho - f) * omega + w_i R
// with every floating-point operation rounded on its own (__dadd_rn /
// __dmul_rn are never contracted into FMA), in that operation order, so the
// result is bit-reproducible against a plain FP64 implementation of the
// method.
//
// Bound by the FP64 pipe (two results per SM and clock: a warp instruction
// every 16 clocks), so every operation that a result does not need is left out:
//  * the weights of a lattice are one weight times powers of two (4/9, 1/9,
//    1/36; 1/3, 1/6, also after rounding), so w_i rho and w_i R take one
//    multiplication each and the others an addition to the exponent, which
//    gives the rounded product wherever it is a normal number (else the
//    products are formed one by one);
//  * a multiplication by omega = 1 (tau = 1) changes nothing and is skipped;
//  * the mass is only summed where it is asked for.
// Two-species Gray-Scott: 99 operations per site instead of 112; one species with
// tau = 1: 38 instead of 54.
#pragma once

#include "lbrd_common.cuh"

namespace lbrd {
namespace f64 {

constexpr int kNT = 128;  // threads of a block; a tile is 128 consecutive sites (row-major)

// Powers of two from the axis weight to the others, per weight class.
template <int Q>
__device__ __forceinline__ constexpr int weight_exp(int c) {
    return Q == 9 ? (c == 0 ? 2 : (c == 1 ? 0 : -2)) : (c == 0 ? 1 : 0);
}
static_assert(Lattice<9>::wc<double>(0) == 4.0 * Lattice<9>::wc<double>(1) &&
                  Lattice<9>::wc<double>(2) == 0.25 * Lattice<9>::wc<double>(1) &&
                  Lattice<5>::wc<double>(0) == 2.0 * Lattice<5>::wc<double>(1),
              "the weights are powers of two apart");

// c[k] = w_k v, rounded, for every weight class k.
template <int Q>
__device__ __forceinline__ void weighted(double v, double (&c)[Lattice<Q>::kClasses]) {
    using L = Lattice<Q>;
    c[1] = __dmul_rn(L::template wc<double>(1), v);
    const int hi = __double2hiint(c[1]), lo = __double2loint(c[1]);
    const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
    // v itself, not the product: w_1 v rounds to zero for the smallest v whose w_0 v does not
    const bool zero = ((__double2hiint(v) & 0x7fffffff) | __double2loint(v)) == 0;
    // exponents 3 .. 2043: the product and its multiples by 1/4 .. 4 are normal; zero stays zero
    const bool plain = e - 3u <= 2040u || zero;
    const unsigned warp = __activemask();
    if (__any_sync(warp, !plain)) {
#pragma unroll
        for (int k = 0; k < L::kClasses; ++k) c[k] = __dmul_rn(L::template wc<double>(k), v);
    } else {
#pragma unroll
        for (int k = 0; k < L::kClasses; ++k)
            if (k != 1) c[k] = __hiloint2double(hi + (zero ? 0 : weight_exp<Q>(k) * (1 << 20)), lo);
    }
}

template <int Q, int S>
__device__ __forceinline__ void site_f64(const StepArgs &a, int x, int y, double *acc) {
    using L = Lattice<Q>;
    // plain loads (no read-only path): the kernel before may still be writing src when this one starts
    const double *src = static_cast<const double *>(a.src);
    double *__restrict__ dst = static_cast<double *>(a.dst);
    const int nx = (int)a.nx, ny = (int)a.ny;
    // pulled rows y + 1, y, y - 1 and columns x + 1, x, x - 1 (periodic), by e + 1
    const int64_t rows[3] = {(int64_t)(y + 1 == ny ? 0 : y + 1) * a.pitch, (int64_t)y * a.pitch,
                             (int64_t)(y == 0 ? ny - 1 : y - 1) * a.pitch};
    const int cols[3] = {x + 1 == nx ? 0 : x + 1, x, x == 0 ? nx - 1 : x - 1};
    double f[S][Q], rho[S];
#pragma unroll
    for (int s = 0; s < S; ++s)
#pragma unroll
        for (int i = 0; i < Q; ++i)
            f[s][i] = src[(int64_t)(s * Q + i) * a.plane + rows[1 + L::ey(i)] + cols[1 + L::ex(i)]];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        double r = f[s][0];
#pragma unroll
        for (int i = 1; i < Q; ++i) r = __dadd_rn(r, f[s][i]);
        rho[s] = r;
    }
    double R[S];
    reaction_f64<S>(a.rkind, a.kappa, a.F, a.k, rho, R);
    double *__restrict__ out = dst + rows[1] + x;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        const double om = a.omega[s];
        double feq[L::kClasses], wr[L::kClasses];
        weighted<Q>(rho[s], feq);
        weighted<Q>(R[s], wr);
        if (om == 1.0) {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                out[(int64_t)(s * Q + i) * a.plane] =
                    __dadd_rn(__dadd_rn(f[s][i], __dsub_rn(feq[L::wclass(i)], f[s][i])), wr[L::wclass(i)]);
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i)
                out[(int64_t)(s * Q + i) * a.plane] = __dadd_rn(
                    __dadd_rn(f[s][i], __dmul_rn(__dsub_rn(feq[L::wclass(i)], f[s][i]), om)), wr[L::wclass(i)]);
        }
        if (a.rho_out) static_cast<double *>(a.rho_out)[(int64_t)s * a.plane + rows[1] + x] = rho[s];
        if (a.mass_out) acc[s] = __dadd_rn(acc[s], rho[s]);
    }
}

// Tiles of 128 consecutive sites of a grid: every lane has a site whatever nx is
// (a row of 100 sites would leave 22 % of the lanes of row-wise tiles idle, at the
// full price in the FP64 pipe).
__host__ __device__ inline int64_t tiles(int64_t nx, int64_t ny) { return (nx * ny + kNT - 1) / kNT; }

template <int Q, int S>
__device__ __forceinline__ void tile_f64(const StepArgs &a, int64_t tile, int thread, double *acc) {
    const unsigned site = (unsigned)tile * kNT + (unsigned)thread;  // sides <= 65535: below 2^32
    const unsigned nx = (unsigned)a.nx, y = site / nx;
    if (y < (unsigned)a.ny) site_f64<Q, S>(a, (int)(site - y * nx), (int)y, acc);
}

}  // namespace f64
}  // namespace lbrd
