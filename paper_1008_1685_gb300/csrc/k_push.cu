// Fused field gather + Boris push + Landau-Lifshitz radiation-reaction kick
// + move + charge-conserving deposit (the particle part of one PIC step).
//
// One CTA per work unit (at most unit_p consecutive particles of one species
// whose cells at the last sort lie in one tile, or in one aligned group or
// half group of sparse tiles holding at most unit_p particles; unit_p is a
// shape of the batch).
// Because cfl < 1 a particle moves less than one cell per step, so k steps
// after the sort every particle of the unit lies in [lo - k, hi + k]; the CTA
// stages the fields of the window [lo - k - 1, hi + k + 2] into shared memory
// (with 4 particles per thread: plain loads into a gather-ready layout; with 2:
// one bulk TMA copy per component, completing on one mbarrier), streams the
// particles (structure of arrays) with 128- or 64-bit evict-first loads and
// stores, and accumulates the unit's current in shared memory.
//
// Deposit: a particle that moves from bin b (cell at x^n) to bin b + d,
// d in {-1, 0, 1}, touches Jy and Jz on at most three nodes and Jx on at most
// two half nodes, all within the stencil anchored at a = min(b, b + d): one
// record of eight values per particle (the 1D Esirkepov split for linear
// shapes: the old bin's share up to the crossing point, the new bin's after
// it).  Determinism: a thread first adds the records of its successive
// particles that share an anchor, in a fixed order; the record is then
// converted to 32-bit fixed point and added to the unit's window in shared
// memory with integer atomics, which hold exact 64-bit sums as pairs of 32-bit
// words (when all lanes of a warp hold the same anchor, as in dense plasma,
// the lanes are first summed exactly by an integer warp reduction).  At the
// end the window is shifted to the 64-bit scale of the accumulators and added
// to global memory with integer atomics.  Integer addition is exact and
// associative, so the result does not depend on the order in which lanes,
// warps or CTAs arrive.
#include "yee.cuh"

namespace picrr {

namespace {

constexpr unsigned FULL = 0xffffffffu;

#ifndef PICRR_THIN_PER_CELL
#define PICRR_THIN_PER_CELL 8
#endif
// Units with fewer particles per cell than this (thinly spread plasma, where
// nearly every lane of a warp holds its own anchor) skip the warp-wide test
// of warp_add altogether: every lane adds its records by itself.
constexpr int kThinPerCell = PICRR_THIN_PER_CELL;

// The unit's current window in shared memory holds exact 64-bit integer sums
// (in the 2^lscale units of the records) as two signed 32-bit words:
// value = hi * 2^32 + lo.  A term t is added with a 32-bit atomic on lo, which
// returns the old word: the addition wrapped iff old and t have one sign and
// old + t the other, and hi then gets that sign.  Every wrap is seen by
// exactly one adder, so the pair always holds the exact sum, in any order.
// Sums stay around zero, so wraps are rare (with lo unsigned, every change of
// the sum's sign was a carry: five more atomics a particle in thin plasma).
// (A 64-bit shared-memory atomic runs at a sixth of the 32-bit rate.)
struct Window {
    int lo[3][WMAX];  // Jx (half nodes), Jy, Jz (nodes)
    int hi[3][WMAX];
};

__device__ __forceinline__ uint32_t win_addr(const Window& w) { return smem_u32(&w.lo[0][0]); }

// Negative if old + t leaves the signed 32-bit range.  (Added as unsigned words, where that is defined.)
__device__ __forceinline__ int win_wrapped(int old, int t) {
    const unsigned o = static_cast<unsigned>(old), a = static_cast<unsigned>(t), now = o + a;
    return static_cast<int>((o ^ now) & (a ^ now));
}
// Adds t to the window word at shared address `addr`; negative if the word wrapped.
__device__ __forceinline__ int win_add(uint32_t addr, int t) {
    int old;
    asm volatile("atom.shared.add.s32 %0, [%1], %2;" : "=r"(old) : "r"(addr), "r"(t) : "memory");
    return win_wrapped(old, t);
}
// The wrap's entry in hi.
__device__ __forceinline__ void win_carry(uint32_t addr, int t) {
    asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr + 3 * WMAX * 4), "r"(t < 0 ? -1 : 1) : "memory");
}

// Position of value q of a stencil record anchored at key: q 0..2 are Jy at
// key+q, 3..5 Jz at key+q-3, 6 and 7 Jx at half nodes key, key+1.
__device__ __forceinline__ int rec_comp(int q) { return q < 3 ? 1 : (q < 6 ? 2 : 0); }
__device__ __forceinline__ int rec_at(int key, int q) { return key + (q < 3 ? q : (q < 6 ? q - 3 : q - 6)); }

// One lane's record added by itself: each value rounded to 32-bit fixed point
// (records are kept in the window's units, |value| < 2^26).  The wraps of its
// values are collected as bits and looked at once: five instructions a value.
// Values that are zero unless a particle crossed a cell boundary (node key + 2,
// half node key + 1) are skipped when all are, and Jz when it is zero (linear
// polarization): adds of zeros to the few words that a warp's lanes share are
// not free (late in the runs of 96 small foils, half of them linear, 217 us a
// push with them, 203 without).
__device__ __forceinline__ void lane_add(int key, const float (&v)[8], uint32_t w) {
    const uint32_t a = w + 4u * key;
    constexpr int at[8] = {4 * WMAX, 4 * (WMAX + 1), 4 * (WMAX + 2), 8 * WMAX, 4 * (2 * WMAX + 1), 4 * (2 * WMAX + 2), 0, 4};
    unsigned wraps = 0u;
    auto add = [&](int q) { wraps = __funnelshift_l(static_cast<unsigned>(win_add(a + at[q], __float2int_rn(v[q]))), wraps, 1); };
    add(0);
    add(1);
    add(6);
    if (v[3] != 0.f || v[4] != 0.f) {
        add(3);
        add(4);
    } else {
        wraps <<= 2;
    }
    if (v[2] != 0.f || v[5] != 0.f || v[7] != 0.f) {
        add(2);
        add(5);
        add(7);
    } else {
        wraps <<= 3;
    }
    if (wraps) {
        constexpr int bit[8] = {7, 6, 2, 4, 3, 1, 5, 0};
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (wraps >> bit[q] & 1u) win_carry(a + at[q], __float2int_rn(v[q]));
    }
}

// One stencil record per lane (key < 0: none).  When every lane holds the
// same anchor (dense plasma), the records are summed exactly in 32-bit fixed
// point (|value| < 2^26 per lane, so the warp sum fits) by one integer warp
// reduction per value and lanes 0..7 add the eight sums (3 % of the large run's
// push against eight adds by lane 0); otherwise every lane adds
// its own record.  (A reduction over lanes grouped by anchor runs once per
// distinct anchor, which costs more than the lanes' own atomics as soon as
// the warp holds two.)
__device__ __forceinline__ void warp_add(int key, const float (&v)[8], uint32_t w, bool vote) {
    const int k0 = __shfl_sync(FULL, key, 0);
    if (vote && __all_sync(FULL, key == k0)) {
        if (k0 >= 0) {
            // lane q (q < 8) adds the warp sum of value q: eight distinct words
            const int lane = threadIdx.x & 31;
            int mine = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int t = __reduce_add_sync(FULL, __float2int_rn(v[q]));
                mine = lane == q ? t : mine;
            }
            if (lane < 8) {
                const uint32_t a = w + 4u * (rec_comp(lane) * WMAX + rec_at(k0, lane));
                if (win_add(a, mine) < 0) win_carry(a, mine);
            }
        }
    } else {
        // (summing the records of neighbouring lanes with one anchor first saves
        // atomics but not time)
        if (key >= 0) lane_add(key, v, w);
    }
}

// Reciprocal square root and quotient for arguments x >= 1 (1 + p^2, 1 + t^2,
// sums of Lorentz factors): the approximate hardware forms with flush of
// subnormal inputs, which never applies to such x, so the subnormal checks of
// the general forms are dropped (2.6 % of the push time on dense foils).
__device__ __forceinline__ float rsqrt_ge1(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float div_ge1(float a, float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return a * y;
}

__device__ __forceinline__ int comp(const int4& a, int j) { return j == 0 ? a.x : j == 1 ? a.y : j == 2 ? a.z : a.w; }
__device__ __forceinline__ float& comp(float4& a, int j) { return j == 0 ? a.x : j == 1 ? a.y : j == 2 ? a.z : a.w; }
__device__ __forceinline__ int comp(const int2& a, int j) { return j == 0 ? a.x : a.y; }
__device__ __forceinline__ float& comp(float2& a, int j) { return j == 0 ? a.x : a.y; }

// A thread takes W consecutive particles per round (one W x 4-byte slot of each
// array).  W = 4: 128-bit loads and stores, fewest instructions per particle,
// for dense foils.  W = 2: 64-bit, fewer registers and so more warps per SM,
// which hides the latency of deposits that scatter over many cells (thinly
// spread particles): 48 registers for 5 CTAs an SM (6 of them, with 40, spill 20
// words: 8 M thinly spread particles 105 us a push against 93).
template <int W>
struct Slot;
template <>
struct Slot<4> {
    using I = int4;
    using F = float4;
    static constexpr int MIN_BLOCKS = 4;
    static __device__ __forceinline__ I pack(const int (&v)[4]) { return make_int4(v[0], v[1], v[2], v[3]); }
    static __device__ __forceinline__ F pack(const float (&v)[4]) { return make_float4(v[0], v[1], v[2], v[3]); }
};
template <>
struct Slot<2> {
    using I = int2;
    using F = float2;
    static constexpr int MIN_BLOCKS = 5;
    static __device__ __forceinline__ I pack(const int (&v)[2]) { return make_int2(v[0], v[1]); }
    static __device__ __forceinline__ F pack(const float (&v)[2]) { return make_float2(v[0], v[1]); }
};

// Shared memory of a CTA: the unit's current window and its field window.  With
// 4 particles per thread (dense foils, many particles per window cell) the
// fields are read with plain loads into a layout made for the gather: per node
// i (Ey, Ey[i+1] - Ey, Ez, Ez[i+1] - Ez) and per half node (Ex, dEx, By, dBy)
// and (Bz, dBz), so that a particle's gather is three loads and five FMAs
// (2 % of the large run's push).  With 2 per thread (thin plasma,
// few particles per cell) the components are copied as they are by bulk TMA,
// and the smaller footprint keeps five CTAs per SM.
template <int W>
struct PushSmem;
template <>
struct PushSmem<4> {
    float4 nd[WMAX];
    float4 hf[WMAX];
    float2 hz[WMAX];
    Window J;
};
template <>
struct PushSmem<2> {
    float F[5][WMAX + 8];  // element 4 is the window's first: room for the halo of the fused update
    Window J;
};

// The Yee update of the fields in F (old, from the element `p0` - 4 of the padded grid on) to the step after,
// for the window's L elements, by all threads of the block; the same arithmetic as field_block.  J: the
// current accumulators of the step, component c's element 0..L at J + c * WMAX.
__device__ __forceinline__ void window_yee(const FieldParams& Q, const RunDev& R, int run, int p0, int L,
                                           float (&F)[5][WMAX + 8], const unsigned long long* J, float (&mur)[8]) {
    const int tid = threadIdx.x, Nx = R.Nx, is = R.is;
    const float* inc = Q.inc + 6 * run;
    const float c = Q.c, hc = Q.hc, fdt = Q.fdt, fpi = R.fp_inv, fph = R.fp_inv * 4294967296.0f;
    const int n0 = p0 - PADF;  // node / half node of the window's element 0 (F[.][4])
    const bool left = n0 <= 0, right = n0 + L >= Nx;  // block-uniform: a wall's node is among elements 0..L
    if (tid < 2 && left) {  // old E of the walls and their neighbours, before they are overwritten
        mur[tid] = F[1 + tid][4 - n0];
        mur[2 + tid] = F[1 + tid][5 - n0];
    }
    if (tid < 2 && right) {
        mur[4 + tid] = F[1 + tid][4 + Nx - n0];
        mur[6 + tid] = F[1 + tid][3 + Nx - n0];
    }
    for (int i = tid + 3; i < L + 5; i += PUSH_T)  // B^{n+1/2} on elements -1..L
        yee_b(F[3][i], F[4][i], F[1][i], F[1][i + 1], F[2][i], F[2][i + 1], hc, n0 + i - 4 == is - 1, inc[0], inc[1]);
    __syncthreads();
    for (int i = tid + 4; i < L + 5; i += PUSH_T) {  // E^{n+1} on elements 0..L
        const int node = n0 + i - 4;
        float ey = F[1][i], ez = F[2][i];
        yee_e(ey, ez, F[3][i - 1], F[3][i], F[4][i - 1], F[4][i], fix_to_float(J[WMAX + i - 4], fpi, fph),
              fix_to_float(J[2 * WMAX + i - 4], fpi, fph), c, fdt, node == is, inc[2], inc[3]);
        const bool inner = node >= 1 && node <= Nx - 1;
        F[1][i] = inner ? ey : 0.f;
        F[2][i] = inner ? ez : 0.f;
    }
    __syncthreads();
    if (left || right) {  // block-uniform
        const float km = (c - 1.f) / (c + 1.f);
        if (tid < 2) {
            float* E = F[1 + tid];
            if (left) E[4 - n0] = yee_mur(mur[2 + tid], E[5 - n0], mur[tid], km);
            if (right) E[4 + Nx - n0] = yee_mur(mur[6 + tid], E[3 + Nx - n0], mur[4 + tid], km);
        }
        __syncthreads();
    }
    for (int i = tid + 4; i < L + 4; i += PUSH_T) {  // B^{n+1} and Ex^{n+1} on elements 0..L-1
        const int node = n0 + i - 4;
        float by = F[3][i], bz = F[4][i];
        yee_b(by, bz, F[1][i], F[1][i + 1], F[2][i], F[2][i + 1], hc, node == is - 1, inc[4], inc[5]);
        const bool in = node >= 0 && node < Nx;
        F[3][i] = in ? by : 0.f;
        F[4][i] = in ? bz : 0.f;
        F[0][i] = in ? fmaf(-fdt, fix_to_float(J[i - 4], fpi, fph), F[0][i]) : 0.f;
    }
}

template <int W, bool FUSED>
__global__ void __launch_bounds__(PUSH_T, Slot<W>::MIN_BLOCKS) k_push_deposit(const PushParams P, const FieldParams Q) {
    using I = typename Slot<W>::I;
    using F = typename Slot<W>::F;
    __shared__ __align__(128) PushSmem<W> sm;
    pdl_release<FUSED>();
    const unsigned phase = *P.phase + P.k;
    [[maybe_unused]] const unsigned before = phase + 5u;  // of the step before
    if constexpr (FUSED) {
        static_assert(W == 2 && sizeof(FieldSmem) <= sizeof(PushSmem<2>), "");
        if (static_cast<int>(blockIdx.x) < Q.nblk) {
            field_block<PUSH_T, true>(Q, before, blockIdx.x, reinterpret_cast<FieldSmem&>(sm));
            return;
        }
    }
    Window& sJ = sm.J;  // the unit's current: Jx (half nodes), Jy, Jz (nodes) of the window
    const uint32_t wJ = win_addr(sJ);
    __shared__ __align__(8) uint64_t bar;
    __shared__ double sred[PUSH_T / 32];

    const int u = FUSED ? blockIdx.x - Q.nblk : blockIdx.x;
    const int run = P.units.run[u];
    if (run < 0) return;  // block-uniform: behind the last unit
    const RunDev& R = P.runs[run];
    if (!R.active) return;
    const int tid = threadIdx.x, lane = tid & 31;
    const int s = P.units.species[u];
    const int par = field_buf(R, FUSED ? before : phase);  // fused: the fields of the step before
    const int start = P.units.start[u], end = P.units.end[u];
    const int lo = P.units.lo[u], hi = P.units.hi[u];
    const int k = P.k;
    // cells [lo - k, hi + k] plus one neighbour left and two right; particles
    // never leave [0, Nx - 1] (frozen ones are skipped), so the window is also
    // clipped to the grid's cells -1 .. Nx + 1, which the guard elements hold
    const int w0 = max(lo - k - 1, -1), w1 = min(hi + k + 3, R.Nx + 2);
    const int p0 = (w0 + PADF) & ~3;
    const int p1 = (w1 + PADF + 3) & ~3;
    const int L = p1 - p0;
    if (L + 4 > WMAX || p0 < 4 || p1 + 4 > R.glen) {  // cannot happen for a valid unit table; never copy out of the arrays
        if (tid == 0) atomicOr(P.status, ST_WINDOW);
        return;
    }

    // the unit's particles are read in slots of W, from the aligned slot before
    // `start` to the aligned slot after `end`; the at most W - 1 particles of
    // each neighbouring unit in those slots are never written here
    const int base = start & ~(W - 1);
    const int nslots = (((end + W - 1) & ~(W - 1)) - base) / W;

    auto clear_window = [&] {
        for (int i = tid; i < L; i += PUSH_T)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                sJ.lo[c][i] = 0;
                sJ.hi[c][i] = 0;
            }
    };
    if constexpr (!FUSED) clear_window();
    const DevSpecies sp = R.sp[s][P.cur];
    if constexpr (W == 2) {
        if (tid == 0) {
            mbar_init(&bar, 1);
            fence_mbar_init();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        pdl_wait<FUSED>();
        if (tid == 0) {
            // fused: with a halo of 4 elements (16 bytes) on each side, which lies inside the padded array, and
            // with the step's current (the window it goes to is not in use yet)
            constexpr int H = FUSED ? 4 : 0;
            const uint32_t bytes = static_cast<uint32_t>(L + 2 * H) * 4u, jbytes = static_cast<uint32_t>(L + 4) * 8u;
            mbar_arrive_expect_tx(&bar, 5u * bytes + (FUSED ? 3u * jbytes : 0u));
#pragma unroll
            for (int c = 0; c < 5; ++c) tma_load_1d(&sm.F[c][4 - H], R.F[par][c] + p0 - H, bytes, &bar);
            if constexpr (FUSED) {
                static_assert(sizeof(Window) >= 3 * WMAX * sizeof(unsigned long long), "");
                unsigned long long* const* J = R.J[current_set(R, before, Q.nsets)];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    tma_load_1d(reinterpret_cast<unsigned long long*>(&sJ) + c * WMAX, J[c] + p0, jbytes, &bar);
            }
        }
        __syncthreads();
    } else {
        const float* const* Fg = R.F[par];
        for (int i = tid; i < L; i += PUSH_T) {
            const int a = p0 + i, b = p0 + (i + 1 < L ? i + 1 : i);  // both within [p0, p1)
            const float ey = __ldg(Fg[1] + a), ez = __ldg(Fg[2] + a), ex = __ldg(Fg[0] + a);
            const float by = __ldg(Fg[3] + a), bz = __ldg(Fg[4] + a);
            sm.nd[i] = make_float4(ey, __ldg(Fg[1] + b) - ey, ez, __ldg(Fg[2] + b) - ez);
            sm.hf[i] = make_float4(ex, __ldg(Fg[0] + b) - ex, by, __ldg(Fg[3] + b) - by);
            sm.hz[i] = make_float2(bz, __ldg(Fg[4] + b) - bz);
        }
    }

    const int rounds = (nslots + PUSH_T - 1) / PUSH_T;
    const float qm = R.qm[s], qw = R.qw[s];
    const float cfl = P.cfl, dt = P.dt, eps = P.eps;
    const float lscale = R.lscale[s];
    const int shift = R.lshift[s];
    const bool rr = s == 0 && R.rr != 0;
    const float hq = 0.5f * qm * dt;
    // the record's factors carry the window's power-of-two scale, so that records
    // are summed in its units (an exact scaling: the same bits as scaling each sum)
    const float jxf = qw / cfl * lscale;  // q w dx / dt
    const float hqw = 0.5f * qw * lscale;

    if constexpr (W == 2) {
        const bool got = mbar_wait_bounded(&bar, 0);
        if (!__syncthreads_and(got)) {
            if (tid == 0) {
                atomicOr(P.status, ST_TIMEOUT);
                mbar_wait_bounded(&bar, 0);  // let the copy land before the CTA exits
            }
            return;
        }
        if constexpr (FUSED) {
            __shared__ float mur[8];
            window_yee(Q, R, run, p0, L, sm.F, reinterpret_cast<const unsigned long long*>(&sJ), mur);
            __syncthreads();
            clear_window();
            __syncthreads();
        }
    } else {
        __syncthreads();
    }

    const bool thin = end - start < kThinPerCell * (hi - lo + 1);  // block-uniform
    // particles can leave the box in this step (block-uniform)
    const bool walls = lo - k <= 0 || hi + k >= R.Nx - 1;
    const unsigned in_unit = static_cast<unsigned>(end - start);
    float rad_h = 0.f, rad_l = 0.f;  // energy radiated by this thread's particles

    // Bound by the instructions issued (225 to 300 a particle).  So the body has no branch on a
    // lane's own state but for the adds: every lane computes its slot's particles (lanes behind
    // the last slot that one's), and those that are not the unit's, frozen or outside the window
    // count for nothing.  us a push with branches -> without: a dense foil of 64 M hot particles
    // 623 -> 540, of cold ones 437 -> 411, 8 M thinly spread ones 107 -> 94.
    for (int r = 0; r < rounds; ++r) {
        const int slot = r * PUSH_T + tid;
        if ((slot & ~31) >= nslots) break;  // the warp has no slot left
        const int b4 = base + W * min(slot, nslots - 1);
        const int rel = base + W * slot - start;
        const I c4 = __ldcs(reinterpret_cast<const I*>(sp.cell + b4));
        F o4 = __ldcs(reinterpret_cast<const F*>(sp.off + b4));
        F x4 = __ldcs(reinterpret_cast<const F*>(sp.px + b4));
        F y4 = __ldcs(reinterpret_cast<const F*>(sp.py + b4));
        F z4 = __ldcs(reinterpret_cast<const F*>(sp.pz + b4));
        // the next round's slots into L2 while this round computes, so that its loads
        // wait on L2 rather than HBM: one bulk (TMA) prefetch per array for the whole
        // CTA, with an evict-first policy (4 % of the large run's push)
        if (tid == 0 && (r + 1) * PUSH_T < nslots) {
            const int n0 = base + W * (r + 1) * PUSH_T;                      // first particle of the next round
            const int n1 = base + W * min((r + 2) * PUSH_T, nslots);         // one past its last
            const int a0 = n0 & ~3, a1 = (n1 + 3) & ~3;                      // 16-byte aligned, within the padded arrays
            const uint32_t bytes = static_cast<uint32_t>(a1 - a0) * 4u;
            uint64_t pol;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
            const void* arrs[5] = {sp.cell + a0, sp.off + a0, sp.px + a0, sp.py + a0, sp.pz + a0};
#pragma unroll
            for (int q = 0; q < 5; ++q)
                asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(arrs[q]), "r"(bytes),
                             "l"(pol)
                             : "memory");
        }
        int cn[W];
        float fo[W], qx[W], qy[W], qz[W];
        bool act[W], all = true;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const int c = comp(c4, j), lb = c + PADF - p0;
            act[j] = static_cast<unsigned>(rel + j) < in_unit && c >= 0 &&
                     static_cast<unsigned>(lb - 1) <= static_cast<unsigned>(L - 4);
            all = all && act[j];
        }
        if (!all) {
#pragma unroll
            for (int j = 0; j < W; ++j) {
                if (act[j]) continue;
                // outside the window: left as it is, reported
                if (static_cast<unsigned>(rel + j) < in_unit && comp(c4, j) >= 0) atomicOr(P.status, ST_WINDOW);
                // whatever the slot holds must not reach the sums as a NaN
                comp(o4, j) = comp(x4, j) = comp(y4, j) = comp(z4, j) = 0.f;
            }
        }
        int rk = -1;  // anchor of this thread's running stencil record
        float rv[8];
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const int c = comp(c4, j);
            const float f = comp(o4, j);
            float px = comp(x4, j), py = comp(y4, j), pz = comp(z4, j);
            const bool a = act[j];
            const int lb = a ? c + PADF - p0 : 1;  // local bin of the particle's cell
            int ka;  // anchor of this particle's stencil record
            float ay, az, w0, w1, w2, dj0, dj1;
            {
                // --- linear gather: nodes (Ey, Ez) and half nodes (Ex, By, Bz)
                const float h = f - 0.5f;
                const int jb = h < 0.f ? lb - 1 : lb;
                const float g = h < 0.f ? h + 1.f : h;
                float e_x, e_y, e_z, b_y, b_z;
                if constexpr (W == 4) {
                    const float4 nd = sm.nd[lb];
                    const float4 hf = sm.hf[jb];
                    const float2 hz = sm.hz[jb];
                    e_y = fmaf(f, nd.y, nd.x);
                    e_z = fmaf(f, nd.w, nd.z);
                    e_x = fmaf(g, hf.y, hf.x);
                    b_y = fmaf(g, hf.w, hf.z);
                    b_z = fmaf(g, hz.y, hz.x);
                } else {
                    const float *sn = &sm.F[0][4] + lb, *sh = &sm.F[0][4] + jb;
                    constexpr int C = WMAX + 8;
                    e_y = (1.f - f) * sn[C] + f * sn[C + 1];
                    e_z = (1.f - f) * sn[2 * C] + f * sn[2 * C + 1];
                    e_x = (1.f - g) * sh[0] + g * sh[1];
                    b_y = (1.f - g) * sh[3 * C] + g * sh[3 * C + 1];
                    b_z = (1.f - g) * sh[4 * C] + g * sh[4 * C + 1];
                }
                // --- Boris step for the Lorentz force (Bx = 0 in 1D)
                const float mx = px + hq * e_x, my = py + hq * e_y, mz = pz + hq * e_z;
                const float ig = rsqrt_ge1(1.f + mx * mx + my * my + mz * mz);
                const float ty = hq * b_y * ig, tz = hq * b_z * ig;
                const float sf = div_ge1(2.f, 1.f + ty * ty + tz * tz);
                const float sy = sf * ty, sz = sf * tz;
                const float ux = mx + my * tz - mz * ty;
                const float uy = my - mx * tz;
                const float uz = mz + mx * ty;
                const float lx = mx + uy * sz - uz * sy + hq * e_x;
                const float ly = my - ux * sz + hq * e_y;
                const float lz = mz + ux * sy + hq * e_z;
                float ign;  // 1 / gamma^{n+1/2}
                if (rr) {
                    // --- Eqs. (estim1, estimgamma): p(n) from p_L and p^{n-1/2}
                    const float bx_ = 0.5f * (lx + px), by_ = 0.5f * (ly + py), bz_ = 0.5f * (lz + pz);
                    const float igb = rsqrt_ge1(1.f + bx_ * bx_ + by_ * by_ + bz_ * bz_);
                    const float vx = bx_ * igb, vy = by_ * igb, vz = bz_ * igb;
                    // f_L = -(E + v x B)
                    const float fx = -(e_x + vy * b_z - vz * b_y);
                    const float fy = -(e_y - vx * b_z);
                    const float fz = -(e_z + vx * b_y);
                    const float av = vx * e_x + vy * e_y + vz * e_z;  // v.E = -v.f_L
                    // gamma^2 [f_L^2 - (v.E)^2] = f_L^2 + |p(n) x f_L|^2 (Lagrange identity),
                    // a sum of squares: no cancellation in single precision
                    const float cx = by_ * fz - bz_ * fy, cy = bz_ * fx - bx_ * fz, cz = bx_ * fy - by_ * fx;
                    const float br = fx * fx + fy * fy + fz * fz + cx * cx + cy * cy + cz * cz;
                    // Eq. (f_r) and Eq. (pertfull): p^{n+1/2} = p_L + dt f_R
                    const float kx = -eps * dt * (fy * b_z - fz * b_y - av * e_x + br * vx);
                    const float ky = -eps * dt * (-fx * b_z - av * e_y + br * vy);
                    const float kz = -eps * dt * (fx * b_y - av * e_z + br * vz);
                    px = lx + kx;
                    py = ly + ky;
                    pz = lz + kz;
                    // gamma(p_L) - gamma(p^{n+1/2}) without cancellation
                    const float qL = 1.f + lx * lx + ly * ly + lz * lz;
                    const float qN = 1.f + px * px + py * py + pz * pz;
                    ign = rsqrt_ge1(qN);
                    const float gL = qL * rsqrt_ge1(qL), gN = qN * ign;
                    // rad_h + rad_l -= de, compensated (Knuth): only rad_l, about 2^-24 of the sum, is rounded at
                    // each particle, so that the units' size changes the tally by 1e-12 at most.  (One addition
                    // in double per round: thin plasma +3 %, a batch of small foils +4 %.)
                    const float dg = div_ge1(kx * (lx + px) + ky * (ly + py) + kz * (lz + pz), gL + gN);
                    const float de = a ? dg : 0.f;
                    const float t = __fsub_rn(rad_h, de), z = __fsub_rn(t, rad_h);
                    rad_l = __fadd_rn(rad_l, __fsub_rn(__fsub_rn(rad_h, __fsub_rn(t, z)), __fadd_rn(de, z)));
                    rad_h = t;
                } else {
                    px = lx;
                    py = ly;
                    pz = lz;
                    ign = rsqrt_ge1(1.f + px * px + py * py + pz * pz);
                }
                // --- move: x^{n+1} = x^n + dt p_x / gamma, in cell units
                const float vxn = px * ign;
                float fn = f + cfl * vxn;
                int d = fn >= 1.f ? 1 : (fn < 0.f ? -1 : 0);
                fn -= static_cast<float>(d);
                const bool edge = fn >= 1.f;  // rounded up to the boundary: same point as (c, 0)
                d = edge ? 0 : d;
                fn = edge ? 0.f : fn;
                int cnew = c + d;
                if (walls) {
                    if (cnew < 0) {  // frozen at x = 0 (sorts under cell 0)
                        fn = 0.f;
                        d = 0;
                        cnew = -1;
                    } else if (cnew >= R.Nx) {  // frozen at x = L (sorts under its last cell Nx-1)
                        fn = 0.f;
                        cnew = -R.Nx;
                    }
                }
                // --- stencil record anchored at a = min(old bin, new bin): Jy, Jz on
                // nodes a..a+2 and Jx on half nodes a, a+1 (Esirkepov for linear shapes).
                // With x0, x1 the old and new positions measured from node a (both in
                // [0, 2)), the linear shape gives node a the weight max(0, 1 - x), node
                // a+2 max(0, x - 1) and node a+1 the rest; Jy and Jz take the weights
                // summed over the two positions (the time-averaged shape, doubled), Jx
                // the charge that crossed half nodes a and a+1.
                {
                    const bool up = d > 0, down = d < 0;
                    ka = down ? lb - 1 : lb;
                    const float x0 = down ? f + 1.f : f, x1 = up ? fn + 1.f : fn;
                    const float s0a = fmaxf(1.f - x0, 0.f), s0b = fmaxf(1.f - x1, 0.f);
                    const float s2a = fmaxf(x0 - 1.f, 0.f), s2b = fmaxf(x1 - 1.f, 0.f);
                    w0 = s0a + s0b;
                    w2 = s2a + s2b;
                    w1 = (2.f - w0) - w2;
                    const float hqi = (a ? hqw : 0.f) * ign;  // (q w / 2) / gamma in the window's units: ay = that times p_y
                    ay = hqi * py;
                    az = hqi * pz;
                    dj0 = s0a - s0b;
                    dj1 = s2b - s2a;
                }
                cn[j] = cnew;
                fo[j] = fn;
            }
            // merge the particle's record into this thread's running record; when
            // its anchor changes, the lane adds the finished record by itself: a warp
            // vote and a warp-wide sum at every change cost more, with 4 particles
            // per thread too (13 % on a dense foil of hot particles, whose anchors
            // change mid-round)
            const float jxa = a ? jxf : 0.f;
            if (j == 0) {
                rk = a ? ka : -1;
                rv[0] = ay * w0;
                rv[1] = ay * w1;
                rv[2] = ay * w2;
                rv[3] = az * w0;
                rv[4] = az * w1;
                rv[5] = az * w2;
                rv[6] = jxa * dj0;
                rv[7] = jxa * dj1;
            } else {
                if (a && rk >= 0 && ka != rk) {
                    lane_add(rk, rv, wJ);
#pragma unroll
                    for (int q = 0; q < 8; ++q) rv[q] = 0.f;
                }
                rk = a ? ka : rk;
                rv[0] = fmaf(ay, w0, rv[0]);
                rv[1] = fmaf(ay, w1, rv[1]);
                rv[2] = fmaf(ay, w2, rv[2]);
                rv[3] = fmaf(az, w0, rv[3]);
                rv[4] = fmaf(az, w1, rv[4]);
                rv[5] = fmaf(az, w2, rv[5]);
                rv[6] = fmaf(jxa, dj0, rv[6]);
                rv[7] = fmaf(jxa, dj1, rv[7]);
            }
            qx[j] = px;
            qy[j] = py;
            qz[j] = pz;
        }
        warp_add(rk, rv, wJ, !thin);
        // with 4 per thread (dense foils), a warp whose particles all stayed in
        // their cells leaves its cell slots as they are: a tenth of the written
        // bytes for most warps of a dense foil (3 % of the large run's push); with
        // 2 per thread (thin, hot plasma, where particles cross cells every step)
        // the vote cost more than it saved
        bool warp_moved = true;
        if constexpr (W == 4) {
            bool moved = false;
#pragma unroll
            for (int j = 0; j < W; ++j) moved = moved || (act[j] && cn[j] != comp(c4, j));
            warp_moved = __any_sync(FULL, moved);
        }
        if (all) {
            if (warp_moved) __stcs(reinterpret_cast<I*>(sp.cell + b4), Slot<W>::pack(cn));
            __stcs(reinterpret_cast<F*>(sp.off + b4), Slot<W>::pack(fo));
            __stcs(reinterpret_cast<F*>(sp.px + b4), Slot<W>::pack(qx));
            __stcs(reinterpret_cast<F*>(sp.py + b4), Slot<W>::pack(qy));
            __stcs(reinterpret_cast<F*>(sp.pz + b4), Slot<W>::pack(qz));
        } else {
#pragma unroll
            for (int j = 0; j < W; ++j) {
                if (!act[j]) continue;
                sp.cell[b4 + j] = cn[j];
                sp.off[b4 + j] = fo[j];
                sp.px[b4 + j] = qx[j];
                sp.py[b4 + j] = qy[j];
                sp.pz[b4 + j] = qz[j];
            }
        }
    }

    // radiated energy: fixed-order sum over the CTA
    if (rr) {
        double v = static_cast<double>(rad_h) + static_cast<double>(rad_l);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
        if (lane == 0) sred[tid >> 5] = v;
    }
    __syncthreads();  // also orders every shared-memory current update before the flush
    if (rr && tid == 0) {
        double t = 0.0;
        for (int w = 0; w < PUSH_T / 32; ++w) t += sred[w];
        P.rad_part[u] += t * static_cast<double>(R.rad_w[s]);  // summed into the tally at the next flush
    }
    const int cset = current_set(R, phase, P.nsets);
    // flush the window: each exact sum shifted from record units to the
    // accumulators' 2^fp units (the run's fixed-point scale keeps it in range)
    for (int i = tid; i < L; i += PUSH_T) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long v = static_cast<long long>(sJ.hi[c][i]) * 4294967296ll + sJ.lo[c][i];
            if (v) atomicAdd(R.J[cset][c] + p0 + i, static_cast<unsigned long long>(v) << shift);
        }
    }
}

}  // namespace

void launch_push(const PushParams& P, const FieldParams& Q, bool fused, int grid, int slot_w, cudaStream_t st, bool pdl) {
    if (grid <= 0) return;
    if (slot_w == 2 && fused)
        launch(k_push_deposit<2, true>, dim3(Q.nblk + grid), PUSH_T, st, pdl, P, Q);
    else if (slot_w == 2)
        launch(k_push_deposit<2, false>, dim3(grid), PUSH_T, st, false, P, Q);
    else
        launch(k_push_deposit<4, false>, dim3(grid), PUSH_T, st, false, P, Q);
}

}  // namespace picrr
