// Division of a list of grids among the warps of a depth-K launch, by rows.
//
// The two-column depth-K kernels walk strips of columns down rows.  Over a list
// the work is one line of rows: strip after strip, every strip its grid's ny
// rows, cut into equal parts, one per worker.  A worker walks its part
// segment by segment (a segment ends with its strip), paying the 2K rows that
// fill the levels once per segment.  Short lists, where that second fill would
// cost more than uneven parts, are cut into bands of one height instead, no
// more bands than workers: 12 uneven grids of sides 64 .. 1024 run at 28.9 us
// per step so and at 30.8 in equal parts, 9 x 512^2 at 15.3 and 16.8 (K = 5).
//
// A worker is a block, whose NW warps walk NW adjacent strips side by side
// (group size NW), or a warp (group size 1).  Strips of consecutive grids of
// equal shape (a "run") are numbered through, so a group may hold the last
// strips of one grid and the first of the next; the last group of a run may be
// partly empty, its remaining warps idle.  Blocks keep the accesses of their
// warps together (the halo columns two strips share are read at about the same
// time, and DRAM sees longer contiguous pieces); single warps lose nothing to
// partly empty groups in lists of uneven grids.
#pragma once

#include "lbrd_kernels.h"

namespace lbrd {

namespace {

// Sites of a list above which the warps of a block meet every four rows (FP32
// D2Q9): the halo columns that two strips share are then read while they are in
// L2.  40 uneven grids of sides up to 2048 (60 M sites): 422 -> 388 us per
// step (K = 5); 256 grids of 255^2: 137 -> 127; 256^2: no change.  Lists that sit
// closer to L2 lose a little instead (9 x 512^2, 2.4 M sites: 16.7 -> 17.3).
constexpr int64_t kLockstepSites = 8 << 20;

// The run of row u, at or after run r: bisection over the runs, which the items
// hold in order.  Each look is a memory latency that depends on the one before, at
// the start of every launch (a run's end stands beside its begin: one look for a
// list of one run).  With a walk from run to run the last workers of 300 grids of
// seven sizes began 85 us late (D2Q9, one species, 60 steps: 1404 us, with bisection
// 357; 120 different grids of 64 .. 183 columns, D2Q5: 1446 and 915).  Out of line:
// inlined, 256 x 256^2 with bf16 deviations took 116.1 us per step instead of 115.0.
__device__ __noinline__ int list_rows_run(const DeepItem *__restrict__ items, int nitems, int64_t u, int r) {
    if (u < items[r].run.end) return r;
    int hi = nitems;
    while (hi - r > 1) {
        const int mid = (r + hi) / 2;
        if (items[mid].run.begin <= u) r = mid;
        else hi = mid;
    }
    return r;
}

// A cut of the line moved to the end of a strip that is at most `slack` rows
// away, so that no worker fills the levels for a few rows of a strip.  r: a run
// at or before the cut's, which it becomes.
__device__ __forceinline__ int64_t list_rows_snap(const DeepItem *__restrict__ items, int nitems, int64_t u,
                                                  int64_t total, int slack, int &r) {
    if (u <= 0 || u >= total) return u;
    r = list_rows_run(items, nitems, u, r);
    const int ny = items[r].run.ny;
    const int at = (int)((u - items[r].run.begin) % ny);
    return at <= slack ? u - at : (ny - at <= slack ? u + (ny - at) : u);
}

// A warp's place in the line: its rows [u, u_end) (in bands: the next band's
// first row and the length of the line), the run of row u and the group size.  Held in shared memory, one per warp, so that it takes no
// registers while a segment's rows are walked.
struct ListWalk {
    int64_t u, u_end;
    int64_t stride;  // list cut into bands: from a worker's band to its next one
    int run, gs;
};

// The place where this warp starts (called by one lane).
template <int NW, int K>
__device__ __forceinline__ void list_rows_begin(const DeepItem *__restrict__ items, int nitems, int64_t total, int w,
                                                ListWalk &walk) {
    const int gs = (int)items[0].gs;
    const int64_t worker = gs == 1 ? (int64_t)blockIdx.x * NW + w : blockIdx.x;
    const int64_t nworkers = gs == 1 ? (int64_t)gridDim.x * NW : gridDim.x;
    const int64_t band = items[0].band;
    walk.gs = gs;
    walk.run = 0;
    if (band > 0) {  // one band per worker (more only if fewer workers run than were planned for)
        walk.u = worker * band;
        walk.u_end = total;
        walk.stride = nworkers * band;
        if (walk.u < total) walk.run = items[list_rows_run(items, nitems, walk.u, 0)].run.item;
        return;
    }
    walk.stride = 0;
    const int64_t rows = total / nworkers;
    const int slack = rows + 1 < 2 * K ? (int)(rows + 1) / 2 : K;
    int r = 0;
    walk.u = list_rows_snap(items, nitems, total * worker / nworkers, total, slack, r);
    walk.run = items[r].run.item;
    walk.u_end = list_rows_snap(items, nitems, total * (worker + 1) / nworkers, total, slack, r);
}

// The next segment: rows [y0, y0 + ly) of strip `strip` of grid `item`;
// `together`: every warp of the block walks a strip of it and the plan asks for
// barriers (block-uniform).  Returns 1, 0 if this warp has no strip in it, or -1 at the end of the part.
// Called by all lanes of the warp.
__device__ __forceinline__ int list_rows_next(const DeepItem *__restrict__ items, int nitems, int w, int lane,
                                              ListWalk &walk, int &item, int &strip, int &y0, int &ly,
                                              bool &together) {
    const volatile ListWalk &wk = walk;
    const int64_t u = wk.u, u_end = wk.u_end;
    if (u >= u_end) return -1;
    const int gs = wk.gs;
    int run = wk.run;
    for (int nx = (int)items[run].next; nx < nitems && items[nx].unit_begin <= u; nx = (int)items[run].next) run = nx;
    const int ny = (int)items[run].a.ny, ns = (int)items[run].nstrips;
    const int64_t local = u - items[run].unit_begin;
    const int height = (int)items[run].height;
    const int group = (int)(local / height);
    y0 = (int)(local - (int64_t)group * height);
    const int64_t stride = wk.stride, most = stride > 0 ? items[0].band : u_end - u;
    ly = ny - y0;
    if (most < ly) ly = (int)most;
    __syncwarp();  // every lane has read the place
    if (lane == 0) {
        walk.u = u + (stride > 0 ? stride : ly);
        walk.run = run;
    }
    __syncwarp();
    together = items[0].lockstep && gs > 1 && group * gs + gs <= (int)items[run].run_strips;
    const int s = gs == 1 ? group : group * gs + w;
    if (s >= (int)items[run].run_strips) return 0;
    item = run + s / ns;
    strip = s - (item - run) * ns;
    return 1;
}

// Fills the runs, the line of rows and the group size (1 or NW) of a list whose
// strips are WO columns wide, for launches of up to nblocks blocks; returns the
// length of the line.
inline int64_t plan_list_rows(DeepItem *items, int n, int K, int WO, int NW, int64_t nblocks) {
    int64_t strip_rows = 0, group_rows = 0, planes = 0;
    int maxny = 1, nruns = 0;
    for (int i = 0; i < n;) {
        int j = i + 1;
        while (j < n && items[j].a.nx == items[i].a.nx && items[j].a.ny == items[i].a.ny) ++j;
        const int64_t ns = (items[i].a.nx + WO - 1) / WO, total = ns * (j - i);
        for (int k = i; k < j; ++k) {
            items[k].nstrips = ns;
            items[k].run_strips = total;
            items[k].next = j;
            planes += items[k].a.plane;
        }
        strip_rows += total * items[i].a.ny;
        group_rows += (total + NW - 1) / NW * items[i].a.ny;
        if (items[i].a.ny > maxny) maxny = (int)items[i].a.ny;
        items[nruns++].run.item = i;
        i = j;
    }
    const int gs = group_rows * NW <= 2 * strip_rows ? NW : 1;
    const int64_t workers = gs == 1 ? nblocks * NW : nblocks, rows = gs == 1 ? strip_rows : group_rows;
    // The smallest band height at which every worker has one band at most, if
    // that takes no more rows per worker than equal shares of the line, most of
    // which cross into a second strip and fill the levels twice.
    int64_t band = 0;
    auto bands_at = [&](int64_t h) {
        int64_t units = 0;
        for (int i = 0; i < n; i = (int)items[i].next)
            units += (items[i].run_strips + gs - 1) / gs * ((items[i].a.ny + h - 1) / h);
        return units;
    };
    if (bands_at(maxny) <= workers) {
        int64_t lo = 1, hi = maxny;
        while (lo < hi) {
            const int64_t mid = (lo + hi) / 2;
            if (bands_at(mid) <= workers) hi = mid;
            else lo = mid + 1;
        }
        if (lo <= rows / workers + 2 * K) band = lo;
    }
    int64_t at = 0;
    for (int r = 0; r < nruns; ++r) {
        const int i = items[r].run.item;
        // a group's place on the line: its rows, or its bands' rows rounded up
        const int64_t height = band > 0 ? (items[i].a.ny + band - 1) / band * band : items[i].a.ny;
        for (int k = i; k < items[i].next; ++k) {
            items[k].gs = gs;
            items[k].lockstep = planes > kLockstepSites;
            items[k].band = band;
            items[k].height = height;
            items[k].unit_begin = at;
        }
        const int64_t begin = at;
        at += (items[i].run_strips + gs - 1) / gs * height;
        items[r].run = {begin, at, i, (int)items[i].a.ny};
    }
    for (int r = nruns; r < n; ++r) items[r].run.begin = INT64_MAX;
    return at;
}

}  // namespace
}  // namespace lbrd
