// Periodic cell sort of the particles of every run of a batch, and the unit
// table built from it.
//
// The sort is a stable counting sort by cell (a particle frozen at a wall
// sorts under its last cell).  It exploits what the push guarantees: a
// particle moves less than one cell per step, so k steps after the last sort
// every particle of unit u has a cell in [lo_u - k, hi_u + k].  It takes three
// launches for all active runs and species of the batch:
//   1. each unit counts its particles per cell of that window; further blocks
//      add the runs' radiated partials into their tallies;
//   2. a block per group of SPAN cells adds the counts of the units whose
//      windows reach into it (they belong to the same or the neighbouring
//      groups of the old table), scans them into the new cell starts and gives
//      every (unit, cell) pair its destination, in unit order.  No scan over
//      blocks is needed: the particles below a group are those of the units
//      wholly below it, which the old order counts, and a part of the counts
//      of the units across its boundary;
//   3. each unit scatters its particles, ranking equal cells in index order
//      (each warp owns a contiguous slice; warp match ranks within a warp and
//      per-warp counts combined in warp order), so the result does not depend
//      on scheduling; further blocks build the new unit table (the tables
//      alternate) from the cell starts: tiles of TILE cells, split into units
//      of at most unit_p particles, except that an aligned group of GROUP
//      consecutive tiles holding at most unit_p particles together forms one
//      unit, or else an aligned half group that does (sparse regions would
//      otherwise give many nearly empty units); when the units are too few to
//      fill the GPU, each is cut into parts of part_p particles, which are the
//      table's entries.
// Every particle is read once and written once; the cell array is read twice
// more for the counts.  In nine launches, with a search for the units of every
// cell and a scan over blocks in between, a sort of a small run took 42 us and
// of thin plasma (8.2M particles) 233 us; in these three 18 and 172 us.
#include <algorithm>
#include <climits>

#include "picrr_internal.cuh"

namespace picrr {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int SORT_T = 256;
constexpr int SCAN_T = 1024;
constexpr int PLAN_T = SPAN;      // threads of the planning kernel: one per cell of a group
constexpr int PLAN_UNITS = 1024;  // units near a group whose bounds are kept in shared memory

// sort key of a stored cell: frozen particles (cell = -1 - k) sort under k
__device__ __forceinline__ int key_of(int c) { return c < 0 ? -1 - c : c; }

__device__ __forceinline__ int groups_of(int Nx) { return (Nx + SPAN - 1) / SPAN; }

// an active run's electron units in the table in use: the first one and their number
__device__ __forceinline__ int2 electron_units(const RunDev& R, int tab) {
    const int32_t* gf = R.group_first[0][tab];
    const int b = gf[0];
    return make_int2(b, gf[groups_of(R.Nx)] - b);
}
// its radiated energy: sum over these units, fixed order (SORT_T threads)
__device__ __forceinline__ void rad_flush_block(const RunDev& R, int2 units, double* part, double* sred) {
    const int b = units.x, n = units.y, t = threadIdx.x;
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (int i = t; i < n; i += 4 * SORT_T) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + q * SORT_T < n) {
                a[q] += part[b + i + q * SORT_T];
                part[b + i + q * SORT_T] = 0.0;
            }
    }
    double v = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if ((t & 31) == 0) sred[t >> 5] = v;
    __syncthreads();
    if (t == 0) {
        double s = 0.0;
        for (int w = 0; w < SORT_T / 32; ++w) s += sred[w];
        R.tally[0] += s;
    }
}

__global__ void __launch_bounds__(SORT_T) k_rad_flush(const RunDev* runs, int tab, double* part) {
    __shared__ double sred[SORT_T / 32];
    const RunDev& R = runs[blockIdx.x];
    if (R.active) rad_flush_block(R, electron_units(R, tab), part, sred);
}

// Sums of grp_n, counted up by count_entries: over each 256 groups, then over each 65536.
__device__ __forceinline__ int sums1(const SortParams& S) { return (S.ngroups + 255) >> 8; }
__device__ __forceinline__ int sums2(const SortParams& S) { return (S.ngroups + 65535) >> 16; }
// cleared by block b of nb (SORT_T threads)
__device__ __forceinline__ void clear_sums(const SortParams& S, int b, int nb) {
    for (int i = b * SORT_T + threadIdx.x; i < sums1(S) + sums2(S); i += nb * SORT_T) S.grp_sum[i] = 0;
}

// ---- 1. per-unit window counts -------------------------------------------------
// Blocks [0, nruns): a run's radiated partials; then a block per unit.
template <bool PDL>
__global__ void __launch_bounds__(SORT_T) k_sort_count(const SortParams S) {
    __shared__ int cnt[SSTR];
    __shared__ double sred[SORT_T / 32];
    pdl_release<PDL>();
    const int u = static_cast<int>(blockIdx.x) - S.nruns;
    if (u < 0) {  // block-uniform
        const RunDev& R = S.runs[blockIdx.x];
        const bool active = R.active;
        const int2 units = active ? electron_units(R, S.tab) : make_int2(0, 0);
        pdl_wait<PDL>();
        clear_sums(S, blockIdx.x, S.nruns);
        if (active) rad_flush_block(R, units, S.rad_part, sred);
        return;
    }
    const int run = S.units.run[u];
    if (run < 0) return;  // block-uniform: behind the last unit
    const RunDev& R = S.runs[run];
    if (!R.active) return;  // a run that ended keeps its particles where they are
    const int s = S.units.species[u];
    const int start = S.units.start[u], end = S.units.end[u];
    const int wb = S.units.lo[u] - S.k;
    const int L = min(S.units.hi[u] + S.k + 1 - wb, SSTR);
    for (int i = threadIdx.x; i < L; i += SORT_T) cnt[i] = 0;
    const int32_t* cell = R.sp[s][S.cur].cell;
    pdl_wait<PDL>();
    __syncthreads();
    constexpr int U = 8;  // loads in flight per thread
    for (int i0 = start; i0 < end; i0 += U * SORT_T) {
        int c[U];
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const int i = i0 + m * SORT_T + threadIdx.x;
            c[m] = i < end ? cell[i] : INT32_MIN;
        }
#pragma unroll
        for (int m = 0; m < U; ++m) {
            if (c[m] == INT32_MIN) continue;
            const int l = key_of(c[m]) - wb;
            // (adds of one are combined by the hardware when lanes share a cell; matching the
            // lanes first took 34 us instead of 17 on thin plasma)
            if (l >= 0 && l < L) atomicAdd(&cnt[l], 1);
            else atomicOr(S.status, ST_WINDOW);
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < L; i += SORT_T) S.cnt[static_cast<size_t>(u) * SSTR + i] = static_cast<uint16_t>(cnt[i]);
}

// ---- 2. cell starts, destinations, entries of the new table -----------------------
// exclusive scan of v over the block (PLAN_T threads)
__device__ __forceinline__ int plan_scan(int v, int* sh, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < PLAN_T / 32 ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        if (lane < PLAN_T / 32) sh[lane] = w;
    }
    __syncthreads();
    *total = sh[PLAN_T / 32 - 1];
    return x - v + (warp > 0 ? sh[warp - 1] : 0);
}

// Table entries of the tiles of a group, from the starts ks[0..cells] of its cells: an
// aligned group of GROUP tiles holding at most unit_p particles is one unit, counted on
// its first tile; otherwise each aligned half group that holds at most unit_p is one;
// otherwise each tile is split on its own.  [a, b): the particles counted on tile t.
__device__ __forceinline__ void tile_range(const int* ks, int cells, int t, int unit_p, int& a, int& b) {
    auto at = [&](int c) { return ks[min(c, cells)]; };
    const int h0 = t / (GROUP / 2) * (SPAN / 2);
    if (at(SPAN) - ks[0] <= unit_p) {
        a = ks[0];
        b = t == 0 ? at(SPAN) : a;
    } else if (at(h0 + SPAN / 2) - at(h0) <= unit_p) {
        a = at(h0);
        b = t % (GROUP / 2) == 0 ? at(h0 + SPAN / 2) : a;
    } else {
        a = at(t * TILE);
        b = at((t + 1) * TILE);
    }
}

// the entries of group j, by the first GROUP threads (ks complete)
__device__ __forceinline__ void count_entries(const SortParams& S, int j, const int* ks, int cells) {
    const int t = threadIdx.x;
    if (t >= 32) return;
    int n = 0;
    if (t < GROUP) {
        int a, b;
        tile_range(ks, cells, t, S.unit_p, a, b);
        n = (b - a + S.part_p - 1) / S.part_p;  // (unit_p is a multiple of part_p)
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) n += __shfl_xor_sync(FULL, n, o);
    if (t == 0) {
        S.grp_n[j] = n;
        if (n) {
            atomicAdd(&S.grp_sum[j >> 8], n);
            atomicAdd(&S.grp_sum[sums1(S) + (j >> 16)], n);
        }
    }
}

// a block per group
template <bool PDL>
__global__ void __launch_bounds__(PLAN_T, 4) k_sort_plan(const SortParams S) {
    __shared__ int sh[PLAN_T / 32];
    __shared__ int ks[SPAN + 1];
    __shared__ int slo[PLAN_UNITS], shi[PLAN_UNITS];
    __shared__ int sbase[2];
    pdl_release<PDL>();
    const int j = blockIdx.x, pair = S.grp_pair[j], s = pair & 1, g = S.grp_at[j], tid = threadIdx.x;
    const RunDev& R = S.runs[pair >> 1];
    const int C0 = g * SPAN, cells = min(SPAN, R.Nx - C0), k = S.k;
    // units of the old table that can reach into the group (k < SPAN)
    const int32_t* gf = R.group_first[s][S.tab];
    const int ua = gf[max(g - 1, 0)], ub = gf[g + 2], nu = ub - ua;
    const bool staged = nu <= PLAN_UNITS;  // else their bounds are read from the table
    for (int i = tid; staged && i < nu; i += PLAN_T) {
        slo[i] = S.units.lo[ua + i] - k;
        shi[i] = S.units.hi[ua + i] + k;
    }
    if (tid < 2) sbase[tid] = 0;
    pdl_wait<PDL>();
    __syncthreads();
    auto lo = [&](int i) { return staged ? slo[i] : S.units.lo[ua + i] - k; };  // windows, both non-decreasing
    auto hi = [&](int i) { return staged ? shi[i] : S.units.hi[ua + i] + k; };
    auto first_reaching = [&](int c) {  // first unit with hi >= c
        int l = 0, r = nu;
        while (l < r) {
            const int m = (l + r) >> 1;
            if (hi(m) >= c) r = m; else l = m + 1;
        }
        return l;
    };
    // (The counts of U units are read together.  With units of 1024 a cell of a dense spot is in the windows of a
    // thousand units: then the last one is searched for, so that no count waits for the bounds of the next unit.
    // One by one, 1.5 M particles in 20 cells took 700 us a sort, now 400.)
    constexpr int U = 4;
    const int key = C0 + tid;
    int tot = 0, u0 = 0, u1 = 0;  // units [u0, u1) cover the cell
    if (tid < cells) {
        u0 = u1 = first_reaching(key);
        int c[U];
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const bool in = u0 + m < nu && lo(u0 + m) <= key;
            c[m] = in ? S.cnt[static_cast<size_t>(ua + u0 + m) * SSTR + (key - lo(u0 + m))] : 0;
            u1 += in ? 1 : 0;
        }
#pragma unroll
        for (int m = 0; m < U; ++m) tot += c[m];
        if (u1 == u0 + U) {
            int r = nu;  // first unit with lo > key
            while (u1 < r) {
                const int m = (u1 + r) >> 1;
                if (lo(m) > key) r = m; else u1 = m + 1;
            }
#pragma unroll 8
            for (int u = u0 + U; u < u1; ++u) tot += S.cnt[static_cast<size_t>(ua + u) * SSTR + (key - lo(u))];
        }
    }
    // particles below the group: those of the units wholly below it, and the counts below it of
    // the units across its start, a warp per unit
    const int uc = first_reaching(C0);  // the same for all threads
    int below = 0;
    for (int i = uc + (tid >> 5); i < nu && lo(i) < C0; i += PLAN_T / 32)
        for (int c = lo(i) + (tid & 31); c < C0; c += 32) below += S.cnt[static_cast<size_t>(ua + i) * SSTR + (c - lo(i))];
    below = __reduce_add_sync(FULL, below);
    if ((tid & 31) == 0 && below) atomicAdd(&sbase[0], below);
    if (tid == 0) sbase[1] = uc < nu ? S.units.start[ua + uc] : (nu > 0 ? S.units.end[ub - 1] : -1);
    int total;
    const int r = plan_scan(tot, sh, &total);
    int below_all = sbase[1];
    if (below_all < 0)  // no unit near: every unit before is below
        below_all = ua > gf[0] ? S.units.end[ua - 1] : 0;
    int at = below_all + sbase[0] + r;
    if (tid < cells) {
        R.keystart[s][key] = at;
        ks[tid] = at;
        if (key == R.Nx - 1) R.keystart[s][R.Nx] = at + tot;
    }
    if (tid == 0) ks[cells] = below_all + sbase[0] + total;
    for (int u = u0; u < u1; u += U) {
        size_t q[U];
        int c[U];
#pragma unroll
        for (int m = 0; m < U; ++m) {
            const bool in = u + m < u1;
            q[m] = in ? static_cast<size_t>(ua + u + m) * SSTR + (key - lo(u + m)) : 0;
            c[m] = in ? S.cnt[q[m]] : 0;
        }
#pragma unroll
        for (int m = 0; m < U; ++m) {
            if (u + m < u1) S.offs[q[m]] = at;
            at += c[m];
        }
    }
    __syncthreads();
    count_entries(S, j, ks, cells);
}

// ---- 3a. the new unit table -------------------------------------------------------
// One block (SORT_T threads) per group: the table index of its first entry is the number of
// entries of the groups before it.  Of these it adds up the sums over 65536 and over 256 of them and
// the rest one by one, so that a block reads at most 512 numbers and those few over 65536, whatever the
// number of groups and of run slots (blocks for every slot, each reading the entries of all of them, made a step
// of one run of 15,000 cells in a batch of 8192 slots 322 us long; it takes 13, and 11 with one slot).
struct FillSmem {
    int ks[SPAN + 1];
    int first[GROUP + 1];
    int red[2];
};
// The table's blocks of a launch: one per group, and one if there is none (the phase advances in any case).
__host__ __device__ __forceinline__ int fill_blocks(const SortParams& S) { return S.ngroups > 0 ? S.ngroups : 1; }

// A group as fill_block needs it: what the launches before do not write, so that it is read before they end.
struct FillGroup {
    int run, s, g, Nx;
    const int32_t* ks;  // starts of its cells
    int32_t* gf;        // the run's group_first of the new table
};
__device__ __forceinline__ FillGroup fill_group(const SortParams& S, int j) {
    FillGroup G{};
    if (j >= S.ngroups) return G;
    const int p = S.grp_pair[j];
    G.g = S.grp_at[j];
    G.run = p >> 1;
    G.s = p & 1;
    const RunDev& R = S.runs[G.run];
    G.Nx = R.Nx;
    G.ks = R.keystart[G.s] + G.g * SPAN;
    G.gf = R.group_first[G.s][S.tab_new];
    return G;
}

__device__ __forceinline__ void fill_block(const SortParams& S, int j, const FillGroup& H, FillSmem& F) {
    const int tid = threadIdx.x, run = H.run, s = H.s, g = H.g, C0 = g * SPAN, cells = min(SPAN, H.Nx - C0);
    if (tid < 2) F.red[tid] = 0;
    if (j < S.ngroups)
        for (int i = tid; i <= cells; i += SORT_T) F.ks[i] = H.ks[i];
    __syncthreads();
    // entries before this group, and in all
    const int n2 = sums2(S);
    const int32_t *sum1 = S.grp_sum, *sum2 = sum1 + sums1(S);
    int before = 0, all = 0;
    for (int i = tid; i < n2; i += SORT_T) {
        const int n = sum2[i];
        all += n;
        before += i < (j >> 16) ? n : 0;
    }
    for (int i = (j >> 16 << 8) + tid; i < (j >> 8); i += SORT_T) before += sum1[i];
    for (int i = (j >> 8 << 8) + tid; i < j; i += SORT_T) before += S.grp_n[i];
    before = __reduce_add_sync(FULL, before);
    all = __reduce_add_sync(FULL, all);
    if ((tid & 31) == 0) {
        atomicAdd(&F.red[0], before);
        atomicAdd(&F.red[1], all);
    }
    __syncthreads();
    all = min(F.red[1], S.max_units);
    if (j == 0 && tid == 0) {
        S.fresh.count[0] = all;
        *S.phase = (*S.phase + S.k) % 6u;
    }
    // behind the last entry (each block of the launch a stretch)
    for (int64_t i = all + static_cast<int64_t>(j) * SORT_T + tid; i < S.max_units;
         i += static_cast<int64_t>(fill_blocks(S)) * SORT_T)
        S.fresh.run[i] = -1;
    if (j >= S.ngroups) return;
    const int base = F.red[0];
    if (tid < 32) {
        int a = 0, b = 0;
        if (tid < GROUP) tile_range(F.ks, cells, tid, S.unit_p, a, b);
        int n = (b - a + S.part_p - 1) / S.part_p, x = n;
#pragma unroll
        for (int o = 1; o < GROUP; o <<= 1) {
            const int y = __shfl_up_sync(FULL, x, o);
            if (tid >= o) x += y;
        }
        if (tid < GROUP) F.first[tid] = x - n;
        if (tid == GROUP - 1) F.first[GROUP] = x;
    }
    __syncthreads();
    const int n = F.first[GROUP], G = groups_of(H.Nx);
    int32_t* gf = H.gf;
    if (tid == 0) gf[g] = base;
    if (g == G - 1 && tid < 3) gf[G + tid] = base + n;
    for (int v = tid; v < n; v += SORT_T) {
        int t = 0;
        while (t + 1 < GROUP && F.first[t + 1] <= v) ++t;
        int a, e;
        tile_range(F.ks, cells, t, S.unit_p, a, e);
        // part i of [a, e); where parts of one unit meet, at a multiple of 4 particles, so
        // that the push's slots, and with them its results, are those of the whole unit
        const int i = v - F.first[t];
        auto cut = [&](int j) {
            const int q = a + j * S.part_p;
            return (j * S.part_p) % S.unit_p ? q & ~3 : q;
        };
        const int b = (i + 1) * S.part_p < e - a ? cut(i + 1) : e;
        a = cut(i);
        auto cell_of = [&](int q) {  // cell of sorted particle q: the last one that starts at or before it
            int l = 0, r = cells;
            while (r - l > 1) {
                const int m = (l + r) >> 1;
                if (F.ks[m] <= q) l = m; else r = m;
            }
            return C0 + l;
        };
        const int u = base + v;
        if (u >= S.max_units) continue;  // cannot happen: the table holds what the runs can need
        S.fresh.run[u] = run;
        S.fresh.species[u] = s;
        S.fresh.start[u] = a;
        S.fresh.end[u] = b;
        S.fresh.lo[u] = cell_of(a);
        S.fresh.hi[u] = cell_of(b - 1);
    }
}

// ---- 3b. stable scatter ----------------------------------------------------------
// Each warp owns one contiguous slice of the unit's particles.  Pass 1 counts
// the slice's particles per cell (warp match; only the warp writes its row);
// the rows are then turned into per-warp destination starts (unit offset plus
// the counts of the warps before, in warp order); pass 2 walks the slice
// again in order and places each particle at its warp's running start plus
// its rank among the lanes with the same cell.  Equal cells therefore keep
// index order, with two block barriers per unit.  (Ranking in pass 1 with the result kept
// in registers, so that nothing in pass 2 waits, and more or fewer blocks an SM and rows in
// flight, were no faster.)
constexpr int SC_W = SORT_T / 32;
constexpr int SC_U = 4;  // slice rows of 32 particles in flight per pass step

__device__ __forceinline__ int window_key(const int32_t* cell, int i, int we, int wb) {
    if (i >= we) return -1;
    const int l = key_of(cell[i]) - wb;
    return (l >= 0 && l < SSTR) ? l : -1;  // out of window cannot happen (counted as an error)
}

// A block per group for the new table, then a block per unit (the table
// holds up to max_units, usually far fewer: behind their empty blocks the others came last,
// 19 us later on thin plasma).
template <bool PDL>
__global__ void __launch_bounds__(SORT_T) k_sort_scatter(const SortParams S) {
    __shared__ int row[SC_W][SSTR];
    pdl_release<PDL>();
    const int u = static_cast<int>(blockIdx.x) - fill_blocks(S);
    if (u < 0) {  // block-uniform
        const FillGroup G = fill_group(S, blockIdx.x);
        pdl_wait<PDL>();
        fill_block(S, blockIdx.x, G, reinterpret_cast<FillSmem&>(row));
        return;
    }
    const int of_run = S.units.run[u];
    if (of_run < 0) return;  // block-uniform: behind the last unit
    const RunDev& R = S.runs[of_run];
    if (!R.active) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = S.units.species[u];
    const int start = S.units.start[u], end = S.units.end[u];
    const int wb = S.units.lo[u] - S.k;
    const DevSpecies src = R.sp[s][S.cur];
    const DevSpecies dst = R.sp[s][1 - S.cur];
    const int per = (end - start + SC_W - 1) / SC_W;
    const int ws = min(end, start + warp * per), we = min(end, ws + per);
    for (int i = tid; i < SC_W * SSTR; i += SORT_T) (&row[0][0])[i] = 0;
    pdl_wait<PDL>();
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    // pass 1: this warp's counts per cell
    for (int i0 = ws; i0 < we; i0 += 32 * SC_U) {  // warp-uniform
        int key[SC_U];
#pragma unroll
        for (int m = 0; m < SC_U; ++m) key[m] = window_key(src.cell, i0 + 32 * m + lane, we, wb);
#pragma unroll
        for (int m = 0; m < SC_U; ++m) {
            const unsigned peers = __match_any_sync(FULL, key[m]);
            if (key[m] >= 0 && lane == __ffs(peers) - 1) row[warp][key[m]] += __popc(peers);
            __syncwarp();
        }
    }
    __syncthreads();
    // per cell of the window: destination start of each warp's particles, in warp order
    const int L = S.units.hi[u] + S.k + 1 - wb;
    for (int l = tid; l < L && l < SSTR; l += SORT_T) {
        int run = S.offs[static_cast<size_t>(u) * SSTR + l];
#pragma unroll
        for (int w = 0; w < SC_W; ++w) {
            const int c = row[w][l];
            row[w][l] = run;
            run += c;
        }
    }
    __syncthreads();
    // pass 2: place the slice's particles in order
    for (int i0 = ws; i0 < we; i0 += 32 * SC_U) {  // warp-uniform
        int cl[SC_U], id[SC_U];
        float of[SC_U], x[SC_U], y[SC_U], z[SC_U];
#pragma unroll
        for (int m = 0; m < SC_U; ++m) {
            const int i = i0 + 32 * m + lane;
            if (i < we) {
                cl[m] = src.cell[i];
                of[m] = src.off[i];
                x[m] = src.px[i];
                y[m] = src.py[i];
                z[m] = src.pz[i];
                id[m] = src.id[i];
            }
        }
#pragma unroll
        for (int m = 0; m < SC_U; ++m) {
            const int i = i0 + 32 * m + lane;
            int key = -1;
            if (i < we) {
                const int l = key_of(cl[m]) - wb;
                key = (l >= 0 && l < SSTR) ? l : -1;
            }
            const unsigned peers = __match_any_sync(FULL, key);
            const int d = key >= 0 ? row[warp][key] + __popc(peers & lt) : -1;
            __syncwarp();
            if (key >= 0 && lane == __ffs(peers) - 1) row[warp][key] += __popc(peers);
            __syncwarp();
            if (d >= 0) {
                dst.cell[d] = cl[m];
                dst.off[d] = of[m];
                dst.px[d] = x[m];
                dst.py[d] = y[m];
                dst.pz[d] = z[m];
                dst.id[d] = id[m];
            }
        }
    }
}

// ---- a table for freshly loaded (already sorted) particles ---------------------------
__device__ __forceinline__ int block_sum_int(int v, int* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    int t = 0;
    if (threadIdx.x == 0)
        for (int w = 0; w < KEY_T / 32; ++w) t += sh[w];
    return t;
}

// exclusive scan of v over the block (KEY_T threads)
__device__ __forceinline__ int block_excl_scan(int v, int* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < KEY_T / 32 ? sh[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        if (lane < KEY_T / 32) sh[lane] = w;
    }
    __syncthreads();
    return x - v + (warp > 0 ? sh[warp - 1] : 0);
}

// exclusive scan of n ints by one block of SCAN_T threads (each thread a
// contiguous range); writes out[0..n) and returns the total
__device__ int block_scan_ranges(const int32_t* in, int32_t* out, int n, int* sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int per = (n + SCAN_T - 1) / SCAN_T;
    const int a = min(n, tid * per), b = min(n, a + per);
    int sum = 0;
    for (int i = a; i < b; ++i) sum += in[i];
    int x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = sh[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;
    }
    __syncthreads();
    int run = x - sum + (warp > 0 ? sh[warp - 1] : 0);
    for (int i = a; i < b; ++i) {
        const int v = in[i];
        out[i] = run;
        run += v;
    }
    const int total = sh[SCAN_T / 32 - 1];
    __syncthreads();
    return total;
}

// ---- scan of the per-block sums, one block per (run, species) --------------
__global__ void __launch_bounds__(SCAN_T) k_scan_blocks(const SortParams S) {
    __shared__ int sh[SCAN_T / 32];
    const RunDev& R = S.runs[blockIdx.x];
    const int s = blockIdx.y;
    if (!R.active) return;
    const int nkb = (R.Nx + KEY_T - 1) / KEY_T;
    const int total = block_scan_ranges(R.blocksum[s], R.blockstart[s], nkb, sh);
    if (threadIdx.x == 0) R.keystart[s][R.Nx] = total;
}

// ---- histogram of already sorted particles (fresh load) -------------------------
// grid (blocks, runs, species); warp-aggregated
__global__ void k_hist(const SortParams S) {
    const RunDev& R = S.runs[blockIdx.y];
    const int s = blockIdx.z;
    if (!R.active) return;
    const int n = R.n[s];
    const int lane = threadIdx.x & 31;
    const int32_t* cell = R.sp[s][S.cur].cell;
    for (int b = blockIdx.x * blockDim.x + (threadIdx.x & ~31); b < n; b += gridDim.x * blockDim.x) {
        const int i = b + lane;
        const int c = i < n ? key_of(cell[i]) : -1;
        const unsigned peers = __match_any_sync(FULL, c);
        if (c >= 0 && c < R.Nx && lane == __ffs(peers) - 1) atomicAdd(&R.keycount[s][c], __popc(peers));
    }
}

__global__ void __launch_bounds__(KEY_T) k_block_sums(const SortParams S) {
    __shared__ int sh[KEY_T / 32];
    const RunDev& R = S.runs[blockIdx.y];
    const int s = blockIdx.z;
    if (!R.active || blockIdx.x * KEY_T >= R.Nx) return;
    const int key = blockIdx.x * KEY_T + threadIdx.x;
    const int v = key < R.Nx ? R.keycount[s][key] : 0;
    const int b = block_sum_int(v, sh);
    if (threadIdx.x == 0) R.blocksum[s][blockIdx.x] = b;
}

__global__ void __launch_bounds__(KEY_T) k_keystart(const SortParams S) {
    __shared__ int sh[KEY_T / 32];
    const RunDev& R = S.runs[blockIdx.y];
    const int s = blockIdx.z;
    if (!R.active || blockIdx.x * KEY_T >= R.Nx) return;
    const int key = blockIdx.x * KEY_T + threadIdx.x;
    const int v = key < R.Nx ? R.keycount[s][key] : 0;
    const int r = block_excl_scan(v, sh);
    if (key < R.Nx) R.keystart[s][key] = R.blockstart[s][blockIdx.x] + r;
}

__global__ void k_zero_keycount(const SortParams S) {
    const RunDev& R = S.runs[blockIdx.y];
    const int s = blockIdx.z;
    if (blockIdx.y == 0 && s == 0) clear_sums(S, blockIdx.x, gridDim.x);
    if (!R.active) return;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < R.Nx + 2; i += gridDim.x * blockDim.x)
        R.keycount[s][i] = 0;
}

// entries of every group, from the cell starts
__global__ void __launch_bounds__(SORT_T) k_group_entries(const SortParams S) {
    __shared__ int ks[SPAN + 1];
    const int j = blockIdx.x, s = S.grp_pair[j] & 1, C0 = S.grp_at[j] * SPAN;
    const RunDev& R = S.runs[S.grp_pair[j] >> 1];
    const int cells = min(SPAN, R.Nx - C0);
    for (int i = threadIdx.x; i <= cells; i += SORT_T) ks[i] = R.keystart[s][C0 + i];
    __syncthreads();
    count_entries(S, j, ks, cells);
}

__global__ void __launch_bounds__(SORT_T) k_fill(const SortParams S) {
    __shared__ FillSmem F;
    fill_block(S, blockIdx.x, fill_group(S, blockIdx.x), F);
}

}  // namespace

void launch_sort(const SortParams& S, cudaStream_t st, int* launches, bool pdl) {
    launch(pdl ? k_sort_count<true> : k_sort_count<false>, dim3(S.max_units + S.nruns), SORT_T, st, pdl, S);
    if (S.ngroups > 0) launch(pdl ? k_sort_plan<true> : k_sort_plan<false>, dim3(S.ngroups), PLAN_T, st, pdl, S);
    launch(pdl ? k_sort_scatter<true> : k_sort_scatter<false>, dim3(S.max_units + fill_blocks(S)), SORT_T, st, pdl, S);
    *launches += 3;
}

void launch_build_units(const SortParams& S, cudaStream_t st, int* launches) {  // S.k == 0
    const dim3 kg(S.kb_max, S.nruns, 2);
    k_zero_keycount<<<dim3(64, S.nruns, 2), 256, 0, st>>>(S);
    k_hist<<<dim3(256, S.nruns, 2), 256, 0, st>>>(S);
    k_block_sums<<<kg, KEY_T, 0, st>>>(S);
    k_scan_blocks<<<dim3(S.nruns, 2), SCAN_T, 0, st>>>(S);
    k_keystart<<<kg, KEY_T, 0, st>>>(S);
    if (S.ngroups > 0) k_group_entries<<<S.ngroups, SORT_T, 0, st>>>(S);
    k_fill<<<fill_blocks(S), SORT_T, 0, st>>>(S);
    *launches += 7;
}

void launch_rad_flush(const RunDev* runs, int nruns, int tab, double* rad_part, cudaStream_t st) {
    k_rad_flush<<<nruns, SORT_T, 0, st>>>(runs, tab, rad_part);
}

// ---- foil loader -------------------------------------------------------------
namespace {
// SplitMix64 (Steele, Lea and Flood 2014): n-th output from state `seed`.
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t n) {
    uint64_t z = seed + n * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

__global__ void k_foil(DevSpecies e, DevSpecies ion, int c0, int ncell, int ppc, uint64_t seed) {
    const int64_t n = static_cast<int64_t>(ncell) * ppc;
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int c = c0 + static_cast<int>(i / ppc);
        const int kk = static_cast<int>(i % ppc);
        const uint64_t r = splitmix64_at(seed, static_cast<uint64_t>(c) * static_cast<uint64_t>(ppc) +
                                                   static_cast<uint64_t>(kk) + 1ull);
        const float off = static_cast<float>(r >> 40) * (1.0f / 16777216.0f);  // exact: 24-bit dyadic
        e.cell[i] = c;
        ion.cell[i] = c;
        e.off[i] = off;
        ion.off[i] = off;
        e.px[i] = e.py[i] = e.pz[i] = 0.f;
        ion.px[i] = ion.py[i] = ion.pz[i] = 0.f;
        e.id[i] = static_cast<int32_t>(i);
        ion.id[i] = static_cast<int32_t>(i);
    }
}
}  // namespace

namespace {
__global__ void k_iota(int32_t* id, int64_t n) {
    for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        id[i] = static_cast<int32_t>(i);
}
}  // namespace

void launch_iota(int32_t* id, int64_t n, cudaStream_t st) {
    const int grid = static_cast<int>(std::min<int64_t>((n + 255) / 256, 152 * 64));
    k_iota<<<grid > 0 ? grid : 1, 256, 0, st>>>(id, n);
}

void launch_foil(DevSpecies e, DevSpecies ion, int c0, int ncell, int ppc, uint64_t seed, cudaStream_t st) {
    const int64_t n = static_cast<int64_t>(ncell) * ppc;
    const int grid = static_cast<int>(std::min<int64_t>((n + 255) / 256, 152 * 64));
    k_foil<<<grid > 0 ? grid : 1, 256, 0, st>>>(e, ion, c0, ncell, ppc, seed);
}

}  // namespace picrr
