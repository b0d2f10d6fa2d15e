// Temporal blocking for the general FP32 step (one to four species, mass-action
// networks): K = 2 or 3 time steps of Eq. relax per pass over HBM.
//
// The scheme of step_f32_deep_kernel.cuh: a warp walks a strip of columns down
// a band of rows, lane l holds one column; level-0 rows are staged per warp by
// cp.async in 16-byte chunks, level m > 1 pulls from level m - 1 carried in
// registers and shifted by shuffles, level K is stored.  2048^2, four species, no
// reaction: K = 3 moves its 1.21 GB per launch in 249 us (0.71 of the measured
// copy rate; one step per launch 186 us); with a ten-step
// network 135 us per step against 229, bound by instruction issue.  A level carries
// (2 x e_iy = +1, 1 x e_iy = 0) rows of every species: 36 registers for four
// D2Q9 species, which bounds K at 3 (the one-step kernels moved 288 bytes per
// site and step; K steps share them).  The output strip is a multiple of four
// columns, so that the staged window always starts at the same place of its
// first 16-byte chunk and fits 36 columns.
//
// Per site the operations of step_general.cu in the same order (sm::radd, the
// network, sm::relax), so K levels give the bits of K single steps.
#include <atomic>

#include "site_math.cuh"
#include "step_f32_deep_kernel.cuh"

namespace lbrd {

namespace {

using namespace sm;

// A mass-action network as kernel parameters: read as constant-bank operands by
// the unrolled evaluation below, so that a step of the network costs a few
// instructions per species and no memory latency.  Measured on four species and
// ten steps at 2048^2, us per step: the shared-memory interpreter of
// site_math.cuh (whose byte loads are shared by the 2 or 4 sites of a thread
// there) 379 at K = 3; one step at a time behind a branch each 159; four steps
// at a time without branches, for the instruction-level parallelism of their
// independent products, 135; that with three copies of a group for its largest
// order 143 and rolled over the groups 161.  The copies matter: the levels'
// evaluations must stay in the instruction cache (two groups 102, three 135).
constexpr int kChunk = 4;
constexpr int kChunks = kMaxReactions / kChunk;
struct NetProg {
    int chunks;                                  // groups of four steps; 0: no reaction
    int max_order[kChunks];                      // largest order in the group
    unsigned ge[3][kMaxSpecies][kMaxReactions];  // ge[e][j]: all ones where the order of species j > e
    float rate[kMaxReactions];
    float change[kMaxSpecies][kMaxReactions];
};

NetProg make_prog(const StepArgs &a) {
    NetProg p{};
    const int nr = a.rkind == kMassAction ? a.net.nr : 0;
    p.chunks = (nr + kChunk - 1) / kChunk;
    for (int r = 0; r < nr; ++r) {
        p.rate[r] = (float)a.net.rate[r];
        for (int j = 0; j < kMaxSpecies; ++j) {
            const int o = a.net.order[r][j];
            for (int e = 0; e < 3; ++e) p.ge[e][j][r] = o > e ? 0xffffffffu : 0u;
            if (o > p.max_order[r / kChunk]) p.max_order[r / kChunk] = o;
            p.change[j][r] = (float)a.net.change[r][j];
        }
    }
    return p;
}

// Steps 4c .. 4c + 3.  A step without a factor that the group tests multiplies by
// 1 (a bit select of rho_j or 1), which changes no value; a step beyond the
// network has rate 0 and no changes.  Third powers are rare and stand behind a
// branch; everything else is one copy per group and level, to stay in the
// instruction cache.
template <int S>
__device__ __forceinline__ void prog_chunk(const NetProg &n, int c, const float (&rho)[S], float (&R)[S]) {
    float p[kChunk];
    const bool cubes = n.max_order[c] > 2;
#pragma unroll
    for (int q = 0; q < kChunk; ++q) p[q] = n.rate[kChunk * c + q];
#pragma unroll
    for (int j = 0; j < S; ++j)
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            if (e == 2 && !cubes) break;
#pragma unroll
            for (int q = 0; q < kChunk; ++q) {
                const unsigned m = n.ge[e][j][kChunk * c + q];
                p[q] = rn_mul(p[q], __uint_as_float((__float_as_uint(rho[j]) & m) | (0x3f800000u & ~m)));
            }
        }
#pragma unroll
    for (int q = 0; q < kChunk; ++q)
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const float k = n.change[s][kChunk * c + q];
            if (k != 0.f) R[s] = rn_fma(k, p[q], R[s]);
        }
}

// R_s(rho) of the network: the operations of sm::network_source in its order
// (p = rate; p *= rho_j, order times, j ascending; R_s = fma(change, p, R_s),
// steps in order, zero changes skipped).
template <int S>
__device__ __forceinline__ void prog_source(const NetProg &n, const float (&rho)[S], float (&R)[S]) {
#pragma unroll
    for (int s = 0; s < S; ++s) R[s] = 0.f;
#pragma unroll
    for (int c = 0; c < kChunks; ++c) {
        if (c >= n.chunks) break;
        prog_chunk<S>(n, c, rho, R);
    }
}

template <int Q, int S>
__device__ __forceinline__ void collide_general(const NetProg &net, const float (&om)[S], float (&f)[S][Q],
                                                float (&rho)[S]) {
    using L = Lattice<Q>;
#pragma unroll
    for (int s = 0; s < S; ++s) {
        float r = f[s][0];
#pragma unroll
        for (int i = 1; i < Q; ++i) r = radd(r, f[s][i]);
        rho[s] = r;
    }
    float R[S];
    prog_source<S>(net, rho, R);
#pragma unroll
    for (int s = 0; s < S; ++s) {  // sm::relax with its per-class products shared
        const float c1 = rn_sub(1.f, om[s]);
        const float t = rn_fma(om[s], rho[s], R[s]);
        float wt[L::kClasses];
#pragma unroll
        for (int c = 0; c < L::kClasses; ++c) wt[c] = rn_mul(L::template wc<float>(c), t);
#pragma unroll
        for (int i = 0; i < Q; ++i) f[s][i] = rn_fma(c1, f[s][i], wt[L::wclass(i)]);
    }
}

template <int K>
struct GenGeom {
    static constexpr int WO = (34 - 2 * K) / 4 * 4;  // output columns per warp
    static constexpr int CW = 36;                    // staged columns
    static constexpr int HL = K - 1;                 // window columns left of the output
    static_assert(WO + 2 * K <= 34 && (HL + 1) % 4 + 34 <= 36 + 3, "the window fits the staged columns");
};

// Three staged rows: row j + 1 is staged once level 1 has read row j - 2, whose slot
// it takes.  That leaves shared memory for 12 warps per SM (186 KB for four D2Q9
// species); with a fourth row (staged an iteration ahead) there are 8, and K = 2
// ran at 167 us per step instead of 142.6.
template <int Q, int S, int K, int NW, int NS, int MINB>
__global__ void __launch_bounds__(NW * 32, MINB)
    step_general_deep_kernel(StepArgs a, const __grid_constant__ NetProg net, int nstrips, int nbands, int band,
                             int emit) {
    using L = Lattice<Q>;
    using G = GenGeom<K>;
    constexpr int SQ = S * Q;
    constexpr int CW = G::CW, WO = G::WO;
    constexpr int kRow = SQ * CW;
    static_assert(NS == 3, "row j + 1 takes the slot of row j - 2");
    constexpr int NCH = CW / 4;
    extern __shared__ __align__(16) float smem[];
    dependent_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float *ring = smem + (size_t)w * NS * kRow;
    const unsigned ring_s = static_cast<unsigned>(__cvta_generic_to_shared(ring));
    float om[S];
    double acc[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
        om[s] = (float)a.omega[s];
        acc[s] = 0.0;
    }
    const int nx = (int)a.nx, ny = (int)a.ny;
    const int nwarps = gridDim.x * NW, units = nstrips * nbands;
    // copy role: chunk cc of planes cq, cq + 3, ... (lanes 27 .. 31 idle)
    const int cq = lane / NCH, cc = lane - NCH * cq;
    for (int u = blockIdx.x * NW + w; u < units; u += nwarps) {
        const int b = u / nstrips, strip = u - b * nstrips;
        const int y0 = b * band;
        const int ly = ny - y0 < band ? ny - y0 : band;
        const int xb = strip * WO - G::HL;  // column of lane 0
        constexpr int o = (4 - (G::HL + 1) % 4) % 4;  // staged column of xb - 1
        const int a0 = xb - 1 - o;                    // first staged column, a multiple of 4
        const int64_t offA = (int64_t)cq * a.plane + (int)wrap_mod(a0 + 4 * cc, nx);
        const int nrows = ly + 2 * K;
        int yl = (int)wrap_mod(y0 - K, ny);
        auto stage = [&](int j, int slot) {
            if (j < nrows && lane < 3 * NCH) {
                const unsigned d = ring_s + (unsigned)(slot * kRow + cq * CW + 4 * cc) * 4u;
                const float *sp = static_cast<const float *>(a.src) + (int64_t)yl * a.pitch + offA;
                int64_t pl3 = 3 * a.plane;
                asm volatile("" : "+l"(pl3));  // no plane multiples kept live across the row loop
#pragma unroll
                for (int r = 0; r < (SQ + 2) / 3; ++r)
                    if (cq + 3 * r < SQ) cp_async16(d + (unsigned)(3 * r * CW * 4), sp + r * pl3);
            }
            yl = yl + 1 == ny ? 0 : yl + 1;
            cp_async_commit();
        };
        stage(0, 0);
        float E0[K - 1][S][Q], P1[K - 1][S][Q], P2[K - 1][S][Q];
#pragma unroll
        for (int m = 0; m < K - 1; ++m)
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int i = 0; i < Q; ++i) E0[m][s][i] = P1[m][s][i] = P2[m][s][i] = 0.f;
        int sl = 0;
        for (int j = 0; j < nrows; ++j) {
            cp_async_wait<0>();  // this lane's copies of row j have landed
            __syncwarp();
            const int s1 = sl == 0 ? NS - 1 : sl - 1, s2 = s1 == 0 ? NS - 1 : s1 - 1;
            // staged rows of iterations j - 2, j - 1, j: pulled with e_iy = +1, 0, -1
            const float *rows0[3] = {ring + s2 * kRow + o + 1 + lane, ring + s1 * kRow + o + 1 + lane,
                                     ring + sl * kRow + o + 1 + lane};
            float f[S][Q], rho[S];
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int i = 0; i < Q; ++i) f[s][i] = rows0[1 - L::ey(i)][(s * Q + i) * CW - L::ex(i)];
            __syncwarp();  // every lane has read row j - 2
            stage(j + 1, sl + 1 == NS ? 0 : sl + 1);
            collide_general<Q, S>(net, om, f, rho);
#pragma unroll
            for (int m = 1; m < K; ++m) {  // level m + 1 from level m (carried index m - 1)
                float h[S][Q];
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        const float v = L::ey(i) < 0 ? f[s][i] : (L::ey(i) == 0 ? E0[m - 1][s][i] : P2[m - 1][s][i]);
                        h[s][i] = L::ex(i) > 0   ? __shfl_up_sync(kFullMask, v, 1)
                                  : L::ex(i) < 0 ? __shfl_down_sync(kFullMask, v, 1)
                                                 : v;
                    }
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int i = 0; i < Q; ++i) {
                        if (L::ey(i) > 0) {
                            P2[m - 1][s][i] = P1[m - 1][s][i];
                            P1[m - 1][s][i] = f[s][i];
                        } else if (L::ey(i) == 0) {
                            E0[m - 1][s][i] = f[s][i];
                        }
                        f[s][i] = h[s][i];
                    }
                collide_general<Q, S>(net, om, f, rho);
            }
            if (j >= 2 * K) {  // level K of row y0 + j - 2K
                const int x = xb + lane;
                if (lane >= G::HL && lane < G::HL + WO && x < nx) {
                    int64_t pl = a.plane;
                    asm volatile("" : "+l"(pl));  // no plane multiples kept live across the row loop
                    const int64_t yx = (int64_t)(y0 + j - 2 * K) * a.pitch + x;
                    float *dp = static_cast<float *>(a.dst) + yx;
                    float *rp = emit ? static_cast<float *>(a.rho_out) : nullptr;
#pragma unroll
                    for (int s = 0; s < S; ++s) {
#pragma unroll
                        for (int i = 0; i < Q; ++i) dp[(s * Q + i) * pl] = f[s][i];
                        if (rp) rp[s * pl + yx] = rho[s];
                        if (a.mass_out) acc[s] += (double)rho[s];
                    }
                }
            }
            sl = sl + 1 == NS ? 0 : sl + 1;
        }
    }
    cp_async_wait<0>();
    if (a.mass_out) block_mass_reduce<S, NW * 32>(acc, a.partials, a.counter, a.mass_out);
}

template <int Q, int S, int K, int NW, int NS, int MINB>
cudaError_t launch_general_deep(const StepArgs &a, cudaStream_t st) {
    if (a.nx % 4 != 0 || a.pitch % 4 != 0) return cudaErrorInvalidValue;
    auto kern = step_general_deep_kernel<Q, S, K, NW, NS, MINB>;
    constexpr size_t smem = (size_t)NW * NS * S * Q * GenGeom<K>::CW * sizeof(float);
    static std::atomic<bool> configured[64] = {};  // per device ordinal (handles on several threads)
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64 || !configured[dev].load()) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        if (dev < 64) configured[dev].store(true);
    }
    const unsigned full = persistent_blocks(kern, NW * 32, INT64_MAX, smem);
    const int64_t nstrips = (a.nx + GenGeom<K>::WO - 1) / GenGeom<K>::WO;
    const int64_t nwarps = (int64_t)full * NW;
    const int64_t nb = choose_bands(2 * K, nstrips, a.ny, nwarps);
    const int64_t band = (a.ny + nb - 1) / nb, nbands = (a.ny + band - 1) / band;
    const int64_t units = nstrips * nbands;
    const unsigned grid = units < nwarps ? (unsigned)((units + NW - 1) / NW) : full;
    return launch_dependent(kern, grid, NW * 32, smem, st, a, make_prog(a), (int)nstrips, (int)nbands, (int)band,
                            a.rho_out != nullptr);
}

template <int K, int NW, int NS, int MINB>
cudaError_t dispatch_general_deep(int Q, int S, const StepArgs &a, cudaStream_t st) {
    if (Q == 9) {
        switch (S) {
            case 1: return launch_general_deep<9, 1, K, NW, NS, MINB>(a, st);
            case 2: return launch_general_deep<9, 2, K, NW, NS, MINB>(a, st);
            case 3: return launch_general_deep<9, 3, K, NW, NS, MINB>(a, st);
            case 4: return launch_general_deep<9, 4, K, NW, NS, MINB>(a, st);
        }
    } else if (Q == 5) {
        switch (S) {
            case 1: return launch_general_deep<5, 1, K, NW, NS, MINB>(a, st);
            case 2: return launch_general_deep<5, 2, K, NW, NS, MINB>(a, st);
            case 3: return launch_general_deep<5, 3, K, NW, NS, MINB>(a, st);
            case 4: return launch_general_deep<5, 4, K, NW, NS, MINB>(a, st);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_step_general_deep(int v, int Q, int S, const StepArgs &a, cudaStream_t st) {
    switch (v) {
        case 0: return dispatch_general_deep<2, 4, 3, 3>(Q, S, a, st);
        case 1: return dispatch_general_deep<2, 4, 3, 2>(Q, S, a, st);
        case 2: return dispatch_general_deep<3, 4, 3, 3>(Q, S, a, st);
        case 3: return dispatch_general_deep<3, 4, 3, 2>(Q, S, a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbrd
