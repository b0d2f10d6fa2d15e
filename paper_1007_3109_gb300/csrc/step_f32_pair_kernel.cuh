// FP32 temporal blocking to depth K with two columns per lane: the depth-K
// scheme of step_f32_deep_kernel.cuh (K time steps of Eq. relax per pass over
// HBM, intermediate levels in registers, a warp walking a strip of columns
// down a band of rows) on a 64-column warp window.
//
// Lane l holds the adjacent columns xb + 2l and xb + 2l + 1.  A pull from the
// left neighbour (e_ix = +1) takes the lane's own first column for its second
// one and the second column of lane l - 1 (a warp shuffle) for its first one;
// e_ix = -1 mirrors it.  So a level costs one shuffle per shifted direction
// for two sites, and each level loses one column per side of a 64-column
// window instead of a 32-column one: with the left halo HL (K rounded up to
// an even count) a warp writes 64 - 2 HL columns, e.g. 56 of 64 at K = 4
// against 26 of 32 for one column per lane.  The price is twice the carried
// registers per level, which bounds K.
//
//   * level 0 (f*(t)): rows staged per warp by cp.async in 16-byte chunks
//     (the row pitch is a multiple of 32): the window's 64 columns start at
//     xb (even), inside the 17 aligned chunks from a0 = xb rounded down to a
//     multiple of 4; lanes 0-15 copy chunk `lane` of the first species' planes
//     (one species: of the even planes), lanes 16-31 chunk `lane - 16` of the
//     second's (the odd planes), lane p < S Q chunk 16 of plane p.  A staged row
//     holds every plane from the grid row its component is pulled from (y - e_iy),
//     so one staged row serves level 1 of one output row and its slot is free
//     again: the ring is the rows in flight and one more, instead of three, and
//     the SM's memory left over is L1, where the halo columns of adjacent strips
//     meet (8192^2, K = 6: 317 -> 295 us per step, with a second row in flight in
//     the same two slots 280; K = 4, 512^2: 3.57 -> 3.30; D2Q5 512^2 2.42 -> 2.07).
//     A launch also starts at the first row level 1 needs, 2K - 2 rows before the
//     first output row instead of 2K.  nx a multiple of 4: no chunk straddles the periodic seam.
//     The ANY form takes any nx: a chunk that reaches past the seam (edge
//     strips only) is copied column by column, a lane per column with its
//     wrapped position from shared memory (with a remainder per copy by the
//     lane that owns the chunk, an edge strip's warp took twice as long per
//     row and every launch waited for it: 4095^2 111 -> 95 us per step); kept apart
//     because the extra paths slow the loop body down even where they never
//     run.  Waits only on the warp's own copy groups.
//   * level 1 pulls the lane's column pair of every plane from the staged row
//     (one 8-byte shared load) and shifts it like the levels
//     above; level m > 1 pulls from level m - 1 carried in registers (the row
//     of this iteration for e_iy = -1, the previous one for e_iy = 0, the one
//     before for e_iy = +1), exactly as the one-column kernel.
//   * level 1 is valid on window columns 1 .. 62 and level m on m .. 63 - m;
//     level K is stored for columns HL .. 63 - HL (8-byte stores; the last
//     column of an odd nx alone in the ANY form), and with `emit` rho(t + K)
//     of level K too.
// Each level collides the lane's two columns together (tb::collide_pair: the
// operations of tb::collide_site per column, one test of the reaction kind
// for both, or none with the kind fixed at compile time): K levels give the
// bits of K single steps.  Units, bands, the periodic wrap and the FP64 mass
// reduction are those of the one-column kernel.
#pragma once

#include "list_rows.cuh"
#include "step_f32_deep_kernel.cuh"

namespace lbrd {

namespace {

// Periodic wrap of a column index in 32-bit arithmetic (inlined, unlike a
// 64-bit remainder, which would put a call into the row loop).
__device__ __forceinline__ int wrap32(int a, int n) {
    const int r = a % n;
    return r < 0 ? r + n : r;
}

__device__ __forceinline__ void cp_async4s(unsigned dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst), "l"(src) : "memory");
}

// Volatile shared-memory loads: a list's grid parameters are read from the
// warp's shared copy where they are used (never hoisted into registers).
__device__ __forceinline__ unsigned long long lds_v64(const void *p) {
    unsigned long long v;
    asm volatile("ld.volatile.shared.u64 %0, [%1];\n" : "=l"(v) : "r"(static_cast<unsigned>(__cvta_generic_to_shared(p))));
    return v;
}
__device__ __forceinline__ unsigned lds_v32(const void *p) {
    unsigned v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(static_cast<unsigned>(__cvta_generic_to_shared(p))));
    return v;
}

// Planes with e_iy = ey, as bits.
template <int Q, int S>
__host__ __device__ constexpr unsigned plane_bits(int ey) {
    unsigned m = 0;
    for (int p = 0; p < S * Q; ++p)
        if (Lattice<Q>::ey(p % Q) == ey) m |= 1u << p;
    return m;
}

template <int K>
struct PairGeom {
    static constexpr int HL = (K + 1) / 2 * 2;  // left (and right) halo columns of the window, even
    static constexpr int WO = 64 - 2 * HL;      // output columns per warp, even
};

// Rows of one level carried in shared memory, private to each lane: the previous
// row's e_iy = 0 components, then the e_iy = +1 components of the two rows before
// (row j takes the place of row j - 2), each a lane's two columns.
template <int Q, int S>
struct PairCarry {
    static constexpr int nE = 3 * S, nP = (Q == 9 ? 3 : 1) * S;
    static constexpr int kWarp = (nE + 2 * nP) * 32;  // float2 per warp and level
};

// ANY: grids of any nx (the seam chunks copied column by column, the last
// column of an odd nx stored alone); otherwise nx must be a multiple of 4.
// RK >= 0: the grid's reaction kind, fixed at compile time.  EA: a row is
// staged as soon as level 1 has read the oldest staged row, whose slot it
// takes: NS rows in flight instead of NS - 1, in the same ring.
// SML: bit m - 1 set: level m's rows are carried in shared memory instead of
// registers (not with PP).  At K = 6 the five carried levels of D2Q9 with two
// species need 180 registers; with level 4 in shared memory (4.6 KB per warp, 24
// eight-byte accesses per row and no moves between rows) the kernel spills 64
// bytes instead of 144 and moves the state once per six steps (8192^2: 280 us per
// step against 319 for K = 5, 2048^2 20.7 / 22.0, 4096^2 71 / 81).  Two levels
// in shared memory take 302 us at 8192^2, K = 7 with three 334.  K = 5 with level 3
// there spills nothing (8192^2 342 -> 319 us).
template <int Q, int S, int K, int NW, int NS, int MINB, bool BATCH, bool PP, bool ANY = false, int RK = -1,
          bool EA = false, int SML = 0>
__global__ void __launch_bounds__(NW * 32, MINB)
    step_pair_kernel(StepArgs a, int64_t nstrips, int64_t nbands, int64_t band, const DeepItem *__restrict__ items,
                     int nitems, int64_t total_units, int emit) {
    using L = Lattice<Q>;
    constexpr int SQ = S * Q;
    constexpr int CW = 68;          // staged columns of a warp row: 17 chunks of four
    constexpr int kRow = SQ * CW;   // one staged row, all planes
    constexpr int P = EA ? NS : NS - 1;  // rows staged ahead of use
    constexpr int F = 2 * K - 2;         // rows that fill the levels before level K's first
    constexpr int HL = PairGeom<K>::HL;
    constexpr int WO = PairGeom<K>::WO;
    constexpr int KC = K > 1 ? K - 1 : 1;
    static_assert(K >= 1 && K <= 8 && P >= 1 && WO > 0, "depth 1 .. 8, a row staged ahead");
    extern __shared__ __align__(16) float smem[];
    dependent_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    float *ring = smem + (size_t)w * NS * kRow;
    const unsigned ring_s = static_cast<unsigned>(__cvta_generic_to_shared(ring));
    using PC = PairCarry<Q, S>;
    static_assert(SML == 0 || !PP, "levels in shared memory: without the pulls-first order");
    constexpr int kSM = __builtin_popcount(SML);
    float2 *carry = reinterpret_cast<float2 *>(smem + (size_t)NW * NS * kRow) + (size_t)w * kSM * PC::kWarp + lane;
    SegArgs g;
    if (!BATCH) {
        load_seg(a, g);
        if (!emit) g.rho_out = nullptr;
    }
    // BATCH: the unit's grid parameters, one copy per warp, read where they
    // are used so that they hold no registers across the row loop (a single
    // grid reads them from the kernel's parameter space)
    __shared__ int wcol_sh[ANY ? NW : 1][ANY ? CW + 2 : 1];
    __shared__ SegArgs seg_sh[BATCH ? NW : 1];
    SegArgs &gs = seg_sh[BATCH ? w : 0];
    auto p_src = [&]() -> const float * {
        if constexpr (BATCH) return reinterpret_cast<const float *>(lds_v64(&gs.src));
        else return static_cast<const float *>(a.src);
    };
    auto p_dst = [&]() -> float * {
        if constexpr (BATCH) return reinterpret_cast<float *>(lds_v64(&gs.dst));
        else return static_cast<float *>(a.dst);
    };
    auto p_rho = [&]() -> float * {
        if constexpr (BATCH) return reinterpret_cast<float *>(lds_v64(&gs.rho_out));
        else return emit ? static_cast<float *>(a.rho_out) : nullptr;
    };
    auto p_pitch = [&]() -> int64_t {
        if constexpr (BATCH) return (int64_t)lds_v64(&gs.pitch);
        else return a.pitch;
    };
    auto p_plane = [&]() -> int64_t {
        if constexpr (BATCH) return (int64_t)lds_v64(&gs.plane);
        else return a.plane;
    };
    // relaxation and reaction constants of the collisions
    auto p_coll = [&]() -> SegArgs {
        if constexpr (BATCH && SML == 0) {
            SegArgs c;
            c.omega[0] = __uint_as_float(lds_v32(&gs.omega[0]));
            c.omega[1] = __uint_as_float(lds_v32(&gs.omega[1]));
            c.rkind = (int)lds_v32(&gs.rkind);
            c.kappa = __uint_as_float(lds_v32(&gs.kappa));
            c.F = __uint_as_float(lds_v32(&gs.F));
            c.k = __uint_as_float(lds_v32(&gs.k));
            return c;
        } else {
            return g;
        }
    };
    // lists of two-species D2Q9 grids and the kernels with a level in shared memory, which are
    // bound by instruction issue: the species of a site packed (lists, 256 x 256^2 at K = 5: 98.0 against
    // 99.4 us per step, 256 x 255^2 137 / 145, 9 x 512^2 16.7 / 17.6; D2Q5 and other single grids gain nothing)
    auto collide = [](const SegArgs &cg, float(&f0)[S][Q], float(&f1)[S][Q], float(&rho0)[S], float(&rho1)[S]) {
        if constexpr ((BATCH || SML) && Q == 9 && S == 2) collide_pair_species<Q, RK>(cg, f0, f1, rho0, rho1);
        else collide_pair<Q, S, RK>(cg, f0, f1, rho0, rho1);
    };
    double acc[S];
#pragma unroll
    for (int s = 0; s < S; ++s) acc[s] = 0.0;
    const int64_t nwarps = (int64_t)gridDim.x * NW;
    const int64_t units = nstrips * nbands;
    // copy role: chunk, and species (two species) or plane parity (one)
    const int cch = lane & 15, cpar = lane >> 4;
    constexpr int kStep = S == 2 ? 1 : 2;  // planes between a lane's copies
    // planes pulled from above and from below (bits)
    constexpr unsigned mUp = plane_bits<Q, S>(1), mDown = plane_bits<Q, S>(-1);
    // BATCH: the warp's place in the list's rows, kept in shared memory like gs
    __shared__ ListWalk walk_sh[BATCH ? NW : 1];
    if constexpr (BATCH) {
        if (lane == 0) list_rows_begin<NW, K>(items, nitems, total_units, w, walk_sh[w]);
        __syncwarp();
    }
    for (int64_t u = (int64_t)blockIdx.x * NW + w; BATCH || u < units; u += nwarps) {
        int64_t strip;
        int y0, ly;
        bool together = false;
        if constexpr (BATCH) {
            int item = 0, st = 0;
            const int more = list_rows_next(items, nitems, w, lane, walk_sh[w], item, st, y0, ly, together);
            if (more < 0) break;
            if (more == 0) continue;
            strip = st;
            load_seg(items[item].a, g);
            if (!emit) g.rho_out = nullptr;
            __syncwarp();  // the previous segment's reads of gs are done
            if (lane == 0) gs = g;
            __syncwarp();
        } else {
            const int64_t b = u / nstrips;
            strip = u - b * nstrips;
            y0 = (int)(b * band);
            ly = (int)a.ny - y0 < (int)band ? (int)a.ny - y0 : (int)band;
        }
        // rows and columns fit 32 bits (sides <= 65535); plane offsets need 64
        const int nx = (int)g.nx, ny = (int)g.ny;
        const int xb = (int)(strip * WO) - HL;  // first window column (even)
        const int a0 = xb - (int)wrap_mod(xb, 4);  // first staged column
        const int o = xb - a0;                     // staged column of xb: 0 or 2
        // this lane's chunks start at columns cA and cB.  ANY: a chunk that reaches past the
        // periodic seam (edge strips only) is copied column by column: chunks [clo, chi) lie
        // inside the grid, the columns of the others have their wrapped positions in wcol_sh,
        // which for a single grid also holds 4 clo and 4 chi (no registers across the row loop)
        const int cA = a0 + 4 * cch, cB = a0 + 64;
        bool edge = false, cleanA = true, cleanB = true;
        int clo4 = 0, chi4 = CW;
        if constexpr (ANY) {
            const int clo = a0 < 0 ? -a0 / 4 : 0;
            int chi = (nx - a0) / 4;
            chi = chi < clo ? clo : (chi > 17 ? 17 : chi);
            edge = clo > 0 || chi < 17;
            clo4 = 4 * clo;
            chi4 = 4 * chi;
            cleanA = cch >= clo && cch < chi;
            cleanB = clo <= 16 && chi > 16;
            __syncwarp();  // the previous unit's reads of wcol are done
            if (edge) {
                for (int q = lane; q < CW; q += 32) wcol_sh[w][q] = wrap32(a0 + q, nx);
                if (lane == 0) {
                    wcol_sh[w][CW] = clo4;
                    wcol_sh[w][CW + 1] = chi4;
                }
            }
            __syncwarp();
        }
        const int64_t offA = (int64_t)(cpar * (S == 2 ? Q : 1)) * g.plane + (ANY ? (cleanA ? cA : 0) : wrap_mod(cA, nx));
        const int64_t offB = (int64_t)(lane < SQ ? lane : 0) * g.plane + (ANY ? (cleanB ? cB : 0) : wrap_mod(cB, nx));
        const int nrows = ly + F;
        int yl = (int)wrap_mod(y0 - K + 1, ny);  // row that is staged next
        auto stage = [&](int j, int slot) {
            if (j < nrows) {
                const int64_t pitch = p_pitch();
                const int yu = yl == 0 ? ny - 1 : yl - 1, yd = yl + 1 == ny ? 0 : yl + 1;
                // the rows that components with e_iy = 0, 1 and -1 are pulled from
                const float *src = p_src();
                const float *row0 = src + (int64_t)yl * pitch, *rowu = src + (int64_t)yu * pitch,
                            *rowd = src + (int64_t)yd * pitch;
                const unsigned d = ring_s + (unsigned)(slot * kRow + cpar * (S == 2 ? Q : 1) * CW + 4 * cch) * 4u;
                int64_t pls = kStep * p_plane();
                asm volatile("" : "+l"(pls));  // no plane multiples kept live across the row loop
                if (!ANY || cleanA) {
#pragma unroll
                    for (int r = 0; r < (SQ + 1) / 2; ++r)
                        if (S == 2 || cpar + 2 * r < SQ) {
                            const int ea = L::ey((S == 2 ? r : 2 * r) % Q), eb = L::ey((S == 2 ? r : 2 * r + 1) % Q);
                            const float *ra = ea > 0 ? rowu : (ea < 0 ? rowd : row0);
                            const float *rb = eb > 0 ? rowu : (eb < 0 ? rowd : row0);
                            cp_async16(d + (unsigned)(kStep * r * CW * 4), (cpar ? rb : ra) + offA + r * pls);
                        }
                }
                if (lane < SQ && cleanB)
                    cp_async16(ring_s + (unsigned)(slot * kRow + lane * CW + 64) * 4u,
                               ((mUp >> lane) & 1 ? rowu : (mDown >> lane) & 1 ? rowd : row0) + offB);
                if constexpr (ANY) {
                    if (edge) {  // warp-uniform: a lane per column, plane by plane
                        const volatile int *wc = wcol_sh[w];
                        const int lo4 = BATCH ? clo4 : wc[CW], hi4 = BATCH ? chi4 : wc[CW + 1], nu = lo4 + CW - hi4;
                        int64_t pl = p_plane();
                        asm volatile("" : "+l"(pl));
                        for (int q = lane; q < nu; q += 32) {
                            const int c = q < lo4 ? q : q - lo4 + hi4;
                            const int x = wc[c];
                            unsigned dc = ring_s + (unsigned)(slot * kRow + c) * 4u;
                            int64_t off = x;  // (unrolled: 16 grids of 2047^2 437 -> 404 us per step)
#pragma unroll
                            for (int s = 0; s < S; ++s) {
#pragma unroll
                                for (int i = 0; i < Q; ++i) {
                                    cp_async4s(dc, (L::ey(i) > 0 ? rowu : (L::ey(i) < 0 ? rowd : row0)) + off);
                                    off += pl;
                                    dc += CW * 4;
                                }
                            }
                        }
                    }
                }
            }
            yl = yl + 1 == ny ? 0 : yl + 1;
            cp_async_commit();
        };
#pragma unroll
        for (int jj = 0; jj < P; ++jj) stage(jj, jj);
        // carried levels 1 .. K - 1, both columns: E0 the previous row's
        // e_iy = 0 components, P1 / P2 the e_iy = +1 components of the
        // previous row and of the one before
        float E0[KC][2][S][Q], P1[KC][2][S][Q], P2[KC][2][S][Q];
#pragma unroll
        for (int m = 0; m < KC; ++m)
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int s = 0; s < S; ++s)
#pragma unroll
                    for (int i = 0; i < Q; ++i) E0[m][c][s][i] = P1[m][c][s][i] = P2[m][c][s][i] = 0.f;
        float sum[S];
#pragma unroll
        for (int s = 0; s < S; ++s) sum[s] = 0.f;
        int sl = 0;
        for (int j = 0; j < nrows; ++j) {
            if constexpr (!EA) stage(j + P, sl + P >= NS ? sl + P - NS : sl + P);
            cp_async_wait<EA ? P - 1 : P>();  // this lane's copies of row j have landed
            __syncwarp();
            const float *row = ring + sl * kRow + o + 2 * lane;  // every component as level 1 pulls it
            float f0[S][Q], f1[S][Q], rho0[S], rho1[S];
            float hp0[KC][S][Q], hp1[KC][S][Q];
            if constexpr (PP) {
#pragma unroll
                for (int m = 1; m < K; ++m)
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int i = 0; i < Q; ++i)
                            if (L::ey(i) >= 0) {
                                const float v0 = L::ey(i) == 0 ? E0[m - 1][0][s][i] : P2[m - 1][0][s][i];
                                const float v1 = L::ey(i) == 0 ? E0[m - 1][1][s][i] : P2[m - 1][1][s][i];
                                hp0[m - 1][s][i] = L::ex(i) > 0   ? __shfl_up_sync(kFullMask, v1, 1)
                                                   : L::ex(i) < 0 ? v1
                                                                  : v0;
                                hp1[m - 1][s][i] = L::ex(i) > 0   ? v0
                                                   : L::ex(i) < 0 ? __shfl_down_sync(kFullMask, v0, 1)
                                                                  : v1;
                                if (L::ey(i) > 0) {
                                    P2[m - 1][0][s][i] = P1[m - 1][0][s][i];
                                    P2[m - 1][1][s][i] = P1[m - 1][1][s][i];
                                }
                            }
            }
            // level 1 from the staged rows
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const float2 v = *reinterpret_cast<const float2 *>(row + (s * Q + i) * CW);
                    f0[s][i] = L::ex(i) > 0 ? __shfl_up_sync(kFullMask, v.y, 1) : (L::ex(i) < 0 ? v.y : v.x);
                    f1[s][i] = L::ex(i) > 0 ? v.x : (L::ex(i) < 0 ? __shfl_down_sync(kFullMask, v.x, 1) : v.y);
                }
            if constexpr (EA) {  // every lane has read row j: its slot takes row j + P
                __syncwarp();
                stage(j + P, sl + P >= NS ? sl + P - NS : sl + P);
            }
            {
                const SegArgs cg = p_coll();
                collide(cg, f0, f1, rho0, rho1);
            }
#pragma unroll
            for (int m = 1; m < K; ++m) {  // level m + 1 from level m (carried index m - 1)
                if constexpr (PP) {
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            if (L::ey(i) > 0) {
                                P1[m - 1][0][s][i] = f0[s][i];
                                P1[m - 1][1][s][i] = f1[s][i];
                            } else if (L::ey(i) == 0) {
                                E0[m - 1][0][s][i] = f0[s][i];
                                E0[m - 1][1][s][i] = f1[s][i];
                            }
                            const float v0 = f0[s][i], v1 = f1[s][i];
                            f0[s][i] = L::ey(i) >= 0 ? hp0[m - 1][s][i]
                                       : L::ex(i) > 0 ? __shfl_up_sync(kFullMask, v1, 1)
                                       : L::ex(i) < 0 ? v1
                                                      : v0;
                            f1[s][i] = L::ey(i) >= 0 ? hp1[m - 1][s][i]
                                       : L::ex(i) > 0 ? v0
                                       : L::ex(i) < 0 ? __shfl_down_sync(kFullMask, v0, 1)
                                                      : v1;
                        }
                } else {
                    float h0[S][Q], h1[S][Q];
                    const bool in_smem = (SML >> (m - 1)) & 1;
                    float2 *cs = carry + __builtin_popcount(SML & ((1 << (m - 1)) - 1)) * PC::kWarp;
                    float2 *cp = cs + (PC::nE + (j & 1) * PC::nP) * 32;
                    int ie = 0, ip = 0;
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            float v0, v1;
                            if (L::ey(i) < 0) {
                                v0 = f0[s][i];
                                v1 = f1[s][i];
                            } else if (in_smem) {
                                const float2 v = L::ey(i) == 0 ? cs[32 * ie++] : cp[32 * ip++];
                                v0 = v.x;
                                v1 = v.y;
                            } else {
                                v0 = L::ey(i) == 0 ? E0[m - 1][0][s][i] : P2[m - 1][0][s][i];
                                v1 = L::ey(i) == 0 ? E0[m - 1][1][s][i] : P2[m - 1][1][s][i];
                            }
                            h0[s][i] = L::ex(i) > 0 ? __shfl_up_sync(kFullMask, v1, 1) : (L::ex(i) < 0 ? v1 : v0);
                            h1[s][i] = L::ex(i) > 0 ? v0 : (L::ex(i) < 0 ? __shfl_down_sync(kFullMask, v0, 1) : v1);
                        }
                    ie = ip = 0;
#pragma unroll
                    for (int s = 0; s < S; ++s)
#pragma unroll
                        for (int i = 0; i < Q; ++i) {
                            if (in_smem) {
                                if (L::ey(i) > 0) cp[32 * ip++] = make_float2(f0[s][i], f1[s][i]);
                                else if (L::ey(i) == 0) cs[32 * ie++] = make_float2(f0[s][i], f1[s][i]);
                            } else if (L::ey(i) > 0) {
                                P2[m - 1][0][s][i] = P1[m - 1][0][s][i];
                                P2[m - 1][1][s][i] = P1[m - 1][1][s][i];
                                P1[m - 1][0][s][i] = f0[s][i];
                                P1[m - 1][1][s][i] = f1[s][i];
                            } else if (L::ey(i) == 0) {
                                E0[m - 1][0][s][i] = f0[s][i];
                                E0[m - 1][1][s][i] = f1[s][i];
                            }
                            f0[s][i] = h0[s][i];
                            f1[s][i] = h1[s][i];
                        }
                }
                const SegArgs cg = p_coll();
                collide(cg, f0, f1, rho0, rho1);
            }
            if (j >= F) {  // level K of row y0 + j - F: window columns HL .. 63 - HL
                const int x = xb + 2 * lane;
                if (lane >= HL / 2 && lane < (HL + WO) / 2 && x < nx) {
                    const int y = y0 + j - F;
                    int64_t pl = p_plane();
                    asm volatile("" : "+l"(pl));  // no plane multiples kept live across the row loop
                    const int64_t yx = (int64_t)y * p_pitch() + x;
                    float *dp = p_dst() + yx;
                    float *rp = p_rho();
                    if (!ANY || x + 1 < nx) {  // both columns (x is even: 8-byte stores)
#pragma unroll
                        for (int s = 0; s < S; ++s) {
#pragma unroll
                            for (int i = 0; i < Q; ++i)
                                *reinterpret_cast<float2 *>(dp + (s * Q + i) * pl) = make_float2(f0[s][i], f1[s][i]);
                            if (rp) *reinterpret_cast<float2 *>(rp + s * pl + yx) = make_float2(rho0[s], rho1[s]);
                            if constexpr (!BATCH) sum[s] += rho0[s] + rho1[s];
                        }
                    } else if constexpr (ANY) {  // the last column of an odd nx
#pragma unroll
                        for (int s = 0; s < S; ++s) {
#pragma unroll
                            for (int i = 0; i < Q; ++i) dp[(s * Q + i) * pl] = f0[s][i];
                            if (rp) rp[s * pl + yx] = rho0[s];
                            if constexpr (!BATCH) sum[s] += rho0[s];
                        }
                    }
                }
            }
            // every lane has read slot j before iteration j + 1 stages into it
            if (BATCH && Q == 9 && together && (j & 3) == 0) __syncthreads();
            else __syncwarp();
            sl = sl + 1 == NS ? 0 : sl + 1;
        }
#pragma unroll
        for (int s = 0; s < S; ++s) acc[s] += (double)sum[s];
    }
    cp_async_wait<0>();
    if constexpr (!BATCH)  // a list's masses come from its densities
        if (a.mass_out) block_mass_reduce<S, NW * 32>(acc, a.partials, a.counter, a.mass_out);
}

template <int Q, int S, int K, int NW, int NS, int MINB, bool BATCH, bool PP = false, bool ANY = false, int RK = -1,
          bool EA = false, int SML = 0>
struct PairKernel {
    // Lists of two D2Q9 species: two blocks per SM, also at the shallow depths whose
    // registers would allow more: with three or four rings L1 has no room for the halo
    // columns (256 x 248^2, us per launch of 2 .. 4 steps: 500, 465, 463 -> 450, 439, 447).
    static constexpr size_t smem =
        NW * ((size_t)NS * S * Q * 68 * sizeof(float) + __builtin_popcount(SML) * PairCarry<Q, S>::kWarp * sizeof(float2));
    static constexpr unsigned kCap = BATCH && S * Q > 10 ? 2 : 0;
    static cudaError_t get(unsigned *full) {
        auto kern = step_pair_kernel<Q, S, K, NW, NS, MINB, BATCH, PP, ANY, RK, EA, SML>;
        static std::atomic<bool> configured[64] = {};
        int dev = 0;
        cudaGetDevice(&dev);
        if (dev < 64 && !configured[dev].load()) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            // (the rest of the SM's memory is L1, where the halo columns of adjacent strips meet)
            if (kCap > 0 && e == cudaSuccess)
                e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)((kCap * (smem + 1024) * 100 + (228 << 10) - 1) / (228 << 10)));
            if (e != cudaSuccess) return e;
            configured[dev].store(true);
        }
        *full = persistent_blocks(kern, NW * 32, INT64_MAX, smem);
        if (kCap > 0 && *full > kCap * sm_count()) *full = kCap * sm_count();
        return cudaSuccess;
    }
};

// Blocks of four warps for a grid: one per SM where that is estimated to be
// faster than as many as fit.  Fewer bands fill the levels fewer times, and a
// warp that has its scheduler to itself walks a row in about 2/3 of the time that
// each of two take (K = 4, deep4vwp_128_minb1_s6, one block per SM against as many as
// fit: 512^2 3.26 us per step with 60 bands, 3.70 with 121; 320 x 256 2.15 / 2.82).
inline unsigned pair_blocks(int K, int64_t nstrips, int64_t ny, unsigned full) {
    const unsigned sms = sm_count();
    if (full <= sms) return full;
    int64_t one = 0, all = 0;
    choose_bands(2 * K - 2, nstrips, ny, (int64_t)sms * 4, &one);
    choose_bands(2 * K - 2, nstrips, ny, (int64_t)full * 4, &all);
    return one * 2 < all * (1 + full / sms) ? sms : full;
}

template <int Q, int S, int K, int NW, int NS, int MINB, bool PP, bool ANY, int RK, bool EA, int SML>
cudaError_t launch_pair_rk(const StepArgs &a, cudaStream_t st) {
    constexpr int WO = PairGeom<K>::WO;
    using PK = PairKernel<Q, S, K, NW, NS, MINB, false, PP, ANY, RK, EA, SML>;
    unsigned full = 0;
    cudaError_t e = PK::get(&full);
    if (e != cudaSuccess) return e;
    const int64_t nstrips = (a.nx + WO - 1) / WO;
    if (NW == 4) full = pair_blocks(K, nstrips, a.ny, full);
    const int64_t nwarps = (int64_t)full * NW;
    const int64_t nb = choose_bands(2 * K - 2, nstrips, a.ny, nwarps);
    const int64_t band = (a.ny + nb - 1) / nb, nbands = (a.ny + band - 1) / band;
    const int64_t units = nstrips * nbands;
    const unsigned grid = units < nwarps ? (unsigned)((units + NW - 1) / NW) : full;
    return launch_dependent(step_pair_kernel<Q, S, K, NW, NS, MINB, false, PP, ANY, RK, EA, SML>, grid,
                            NW * 32, PK::smem, st, a, nstrips, nbands, band, nullptr, 0, 0, a.rho_out != nullptr);
}

// Two-species Gray-Scott grids run the form with the reaction fixed at
// compile time (no test of the kind in the row loop); the others test it.
template <int Q, int S, int K, int NW, int NS, int MINB, bool PP, bool ANY = false, bool EA = false, int SML = 0>
cudaError_t launch_pair(const StepArgs &a, cudaStream_t st) {
    if ((!ANY && a.nx % 4 != 0) || a.pitch % 4 != 0) return cudaErrorInvalidValue;
    if constexpr (S == 2)
        if (a.rkind == kGrayScott) return launch_pair_rk<Q, S, K, NW, NS, MINB, PP, ANY, kGrayScott, EA, SML>(a, st);
    return launch_pair_rk<Q, S, K, NW, NS, MINB, PP, ANY, -1, EA, SML>(a, st);
}

}  // namespace
}  // namespace lbrd
