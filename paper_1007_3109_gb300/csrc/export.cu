// Read-out kernels: distributions and densities to packed FP64, and the FP64
// global sum of the densities (sum_x rho_s, the mass diagnostic; conserved
// when R = 0 because sum_i f_eq = rho and sum_i w_i = 1, Eq. equili).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "lbrd_kernels.h"
#include "lb_rd.h"

namespace lbrd {

namespace {

// float to double, exactly, on the integer pipe (the FP64 pipe converts two
// values per SM and clock: 0.21 ms for the 1.3e8 densities of 8192^2, two
// species): the exponent rebased by 1023 - 127, the mantissa moved up 29 bits;
// subnormals normalised, infinities and NaN by their exponent.
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(float v) {
    const unsigned b = __float_as_uint(v), sign = b & 0x80000000u;
    unsigned mag = b & 0x7fffffffu, base = 0x38000000u;
    if (mag - 0x00800000u >= 0x7f000000u) {  // zero, subnormal, infinite or NaN
        if (mag >= 0x7f800000u) {
            base = 0x70000000u;  // exponent 255 -> 2047
        } else if (mag == 0u) {
            base = 0u;
        } else {
            const int up = __clz((int)mag) - 8;  // the leading one to bit 23, which then adds 1 to the exponent
            mag <<= up;
            base -= (unsigned)up << 20;
        }
    }
    return __hiloint2double((int)(sign | ((mag >> 3) + base)), (int)(mag << 29));
}

template <typename T>
struct Pair;
template <>
struct Pair<float> {
    using type = float2;
};
template <>
struct Pair<double> {
    using type = double2;
};

// Two consecutive columns of a packed output row; `vec`: the rows start on
// 16-byte boundaries.
__device__ __forceinline__ void store_pair(double *p, double a, double b, bool both, bool vec) {
    if (both && vec) {
        *reinterpret_cast<double2 *>(p) = make_double2(a, b);
    } else {
        p[0] = a;
        if (both) p[1] = b;
    }
}

bool pairs_aligned(const double *out, int64_t nx) { return nx % 2 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0; }

// Full-precision state: plane p = s * Q + i, value at [p][y][pitch]; two columns
// per thread (the pitch is a multiple of 32, so a pair never leaves its row).
template <typename T>
__global__ void export_plain_kernel(const T *state, int64_t nx, int64_t ny, int64_t pitch, double *out, bool vec) {
    const int64_t x = 2 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
    const int64_t row = (int64_t)blockIdx.z * ny + blockIdx.y;
    if (x >= nx) return;
    const auto v = *reinterpret_cast<const typename Pair<T>::type *>(state + row * pitch + x);
    store_pair(out + row * nx + x, to_double(v.x), to_double(v.y), x + 1 < nx, vec);
}

// Reduced state, per species: plane 0 = rho* (float), planes 1..Q-1 the
// 16-bit deviations g_i; f*_i = w_i rho* + g_i, g_0 = -sum_{i>=1} g_i.
template <int Q, typename H>
__global__ void export_half_kernel(const char *state, int64_t nx, int64_t ny, int64_t pitch, int S, double *out) {
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t y = blockIdx.y;
    const int s = blockIdx.z;
    if (x >= nx) return;
    const int64_t plane = ny * pitch;
    const size_t species_bytes = (size_t)plane * (4 + 2 * (Q - 1));
    const char *base = state + (size_t)s * species_bytes;
    const float rs = reinterpret_cast<const float *>(base)[y * pitch + x];
    const H *g = reinterpret_cast<const H *>(base + (size_t)plane * 4);
    float gs[Q];
    float sum = 0.f;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
        gs[i] = (float)g[(int64_t)(i - 1) * plane + y * pitch + x];
        sum = rn_add(sum, gs[i]);
    }
    gs[0] = -sum;
#pragma unroll
    for (int i = 0; i < Q; ++i)
        out[(((int64_t)s * Q + i) * ny + y) * nx + x] = (double)rn_fma(weight<Q, float>(i), rs, gs[i]);
}

// Densities to packed FP64 and their global FP64 sum, in one pass over the
// density cache.  A block of 256 threads covers 2 bx columns (two per thread) and
// 256 / bx rows, kReadRows times, and walks such tiles with a grid stride, so
// that at most 8 blocks per SM leave partial sums for the last block to add.
// Bound by HBM with the output (8192^2, two species: 1.61 GB in 0.28 ms; the
// separate kernels of one value per thread took 0.41 + 0.72 ms, the second with
// 32768 partial sums per species read by one block) and by the FP64 additions
// (two per SM and clock) without it.
constexpr int kReadNT = 256;
constexpr int kReadRows = 4;

template <typename T, int S>
__global__ void __launch_bounds__(kReadNT) readout_kernel(const T *__restrict__ rho, int64_t nx, int64_t ny,
                                                          int64_t pitch, double *__restrict__ out, bool vec,
                                                          int64_t tiles_x, int64_t ntiles, double *partials,
                                                          unsigned int *counter, double *mass) {
    using P = typename Pair<T>::type;
    double acc[S];
#pragma unroll
    for (int s = 0; s < S; ++s) acc[s] = 0.0;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t ty = t / tiles_x;
        const int64_t x = 2 * ((t - ty * tiles_x) * blockDim.x + threadIdx.x);
        const int64_t y0 = ty * (kReadRows * blockDim.y) + threadIdx.y;
        if (x >= nx) continue;
        P v[kReadRows][S];
#pragma unroll
        for (int r = 0; r < kReadRows; ++r) {
            const int64_t y = y0 + (int64_t)r * blockDim.y;
            if (y < ny) {
#pragma unroll
                for (int s = 0; s < S; ++s)
                    v[r][s] = *reinterpret_cast<const P *>(rho + ((int64_t)s * ny + y) * pitch + x);
            }
        }
#pragma unroll
        for (int r = 0; r < kReadRows; ++r) {
            const int64_t y = y0 + (int64_t)r * blockDim.y;
            if (y < ny) {
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const double a = to_double(v[r][s].x), b = to_double(v[r][s].y);
                    if (out) store_pair(out + ((int64_t)s * ny + y) * nx + x, a, b, x + 1 < nx, vec);
                    if (mass) {
                        acc[s] += a;
                        if (x + 1 < nx) acc[s] += b;
                    }
                }
            }
        }
    }
    if (mass) block_mass_reduce<S, kReadNT>(acc, partials, counter, mass);
}

// Threads of a readout block along x: 32 .. 256, no wider than the row needs.
int readout_bx(int64_t nx) {
    int bx = 32;
    while (bx < kReadNT && 2 * bx < nx) bx *= 2;
    return bx;
}

int64_t readout_tiles(int64_t nx, int64_t ny, int64_t *tiles_x) {
    const int bx = readout_bx(nx), by = kReadNT / bx;
    *tiles_x = (nx + 2 * bx - 1) / (2 * bx);
    return *tiles_x * ((ny + kReadRows * by - 1) / (kReadRows * by));
}

template <typename T, int S>
cudaError_t launch_readout_s(const T *rho, int64_t nx, int64_t ny, int64_t pitch, double *out, double *partials,
                             unsigned int *counter, double *mass, cudaStream_t st) {
    int64_t tiles_x = 0;
    const int64_t ntiles = readout_tiles(nx, ny, &tiles_x);
    const int bx = readout_bx(nx);
    const unsigned grid = persistent_blocks(readout_kernel<T, S>, kReadNT, ntiles);
    readout_kernel<T, S><<<grid, dim3(bx, kReadNT / bx), 0, st>>>(rho, nx, ny, pitch, out, pairs_aligned(out, nx),
                                                                  tiles_x, ntiles, partials, counter, mass);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_readout_t(int S, const T *rho, int64_t nx, int64_t ny, int64_t pitch, double *out,
                             double *partials, unsigned int *counter, double *mass, cudaStream_t st) {
    switch (S) {
        case 1: return launch_readout_s<T, 1>(rho, nx, ny, pitch, out, partials, counter, mass, st);
        case 2: return launch_readout_s<T, 2>(rho, nx, ny, pitch, out, partials, counter, mass, st);
        case 3: return launch_readout_s<T, 3>(rho, nx, ny, pitch, out, partials, counter, mass, st);
        case 4: return launch_readout_s<T, 4>(rho, nx, ny, pitch, out, partials, counter, mass, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

size_t state_plane_bytes(int prec, int Q, int S, int64_t ny, int64_t pitch) {
    const size_t plane = (size_t)ny * (size_t)pitch;
    switch (prec) {
        case LB_RD_FP64: return plane * 8 * Q * S;
        case LB_RD_FP32: return plane * 4 * Q * S;
        default: return plane * (4 + 2 * (Q - 1)) * S;
    }
}

cudaError_t launch_export(int prec, int Q, int S, const void *state, int64_t nx, int64_t ny, int64_t pitch,
                          double *out, cudaStream_t st) {
    const dim3 b(256);
    if (prec == LB_RD_FP64 || prec == LB_RD_FP32) {
        const dim3 g((unsigned)((nx + 511) / 512), (unsigned)ny, (unsigned)(Q * S));
        const bool vec = pairs_aligned(out, nx);
        if (prec == LB_RD_FP64)
            export_plain_kernel<double><<<g, b, 0, st>>>(static_cast<const double *>(state), nx, ny, pitch, out, vec);
        else
            export_plain_kernel<float><<<g, b, 0, st>>>(static_cast<const float *>(state), nx, ny, pitch, out, vec);
        return cudaGetLastError();
    }
    const dim3 g((unsigned)((nx + 255) / 256), (unsigned)ny, (unsigned)S);
    const char *p = static_cast<const char *>(state);
    if (prec == LB_RD_FP32_BF16DEV) {
        if (Q == 9) export_half_kernel<9, __nv_bfloat16><<<g, b, 0, st>>>(p, nx, ny, pitch, S, out);
        else export_half_kernel<5, __nv_bfloat16><<<g, b, 0, st>>>(p, nx, ny, pitch, S, out);
    } else {
        if (Q == 9) export_half_kernel<9, __half><<<g, b, 0, st>>>(p, nx, ny, pitch, S, out);
        else export_half_kernel<5, __half><<<g, b, 0, st>>>(p, nx, ny, pitch, S, out);
    }
    return cudaGetLastError();
}

// One per block of the read-out: no more than fit the device, whatever the grid.
size_t mass_partials_needed(int64_t nx, int64_t ny) {
    int64_t tiles_x = 0;
    return (size_t)std::min<int64_t>(readout_tiles(nx, ny, &tiles_x), max_persistent_blocks());
}

cudaError_t launch_readout(int prec, int S, const void *rho, int64_t nx, int64_t ny, int64_t pitch, double *out,
                           double *partials, unsigned int *counter, double *mass, cudaStream_t st) {
    if (prec == LB_RD_FP64)
        return launch_readout_t<double>(S, static_cast<const double *>(rho), nx, ny, pitch, out, partials, counter,
                                        mass, st);
    return launch_readout_t<float>(S, static_cast<const float *>(rho), nx, ny, pitch, out, partials, counter, mass, st);
}

}  // namespace lbrd
