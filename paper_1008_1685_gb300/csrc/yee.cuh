// The 1D Yee update of one step, as device code shared by the Yee kernel and by the
// push kernel (which updates the fields of its own window when the two are fused):
//   B^{n+1/2} = B^n - (dt/2) curl E^n,
//   E^{n+1}   = E^n + dt (curl B^{n+1/2} - J^{n+1/2}),
//   B^{n+1}   = B^{n+1/2} - (dt/2) curl E^{n+1},
// with the current of this step, total-field / scattered-field laser injection
// (incident values evaluated in double precision by the host for each step) and
// first-order Mur ends.  Every multiply-add is written out, so that both kernels
// give the same bits.
#pragma once

#include "picrr_internal.cuh"

namespace picrr {

// 64-bit fixed-point accumulator (2^fp units) to float from its two 32-bit
// halves (32-bit conversions only): hi * 2^(32-fp) + lo * 2^-fp.
__device__ __forceinline__ float fix_to_float(unsigned long long a, float lo_scale, float hi_scale) {
    const int hi = static_cast<int>(static_cast<long long>(a) >> 32);
    const unsigned lo = static_cast<unsigned>(a & 0xffffffffull);
    return fmaf(static_cast<float>(hi), hi_scale, static_cast<float>(lo) * lo_scale);
}

// Half a step of B on half node j between nodes with E (ey0, ez0) and (ey1, ez1); ay and
// az: incident E on the scattered side of the source plane (j == is - 1).
__device__ __forceinline__ void yee_b(float& by, float& bz, float ey0, float ey1, float ez0, float ez1, float hc, bool src,
                                      float ay, float az) {
    by = fmaf(hc, ez1 - ez0, by);
    bz = fmaf(-hc, ey1 - ey0, bz);
    if (src) {
        bz = fmaf(hc, ay, bz);
        by = fmaf(-hc, az, by);
    }
}

// E of one step on an interior node between half nodes with B^{n+1/2} (by0, bz0) and
// (by1, bz1); ay and az: incident B on the total side (node is).
__device__ __forceinline__ void yee_e(float& ey, float& ez, float by0, float by1, float bz0, float bz1, float jy, float jz,
                                      float c, float fdt, bool src, float ay, float az) {
    ey = fmaf(-fdt, jy, fmaf(-c, bz1 - bz0, ey));
    ez = fmaf(-fdt, jz, fmaf(c, by1 - by0, ez));
    if (src) {
        ey = fmaf(c, ay, ey);
        ez = fmaf(c, az, ez);
    }
}

// First-order Mur end: the new E on the wall from its neighbour's old and new E and its own old E.
__device__ __forceinline__ float yee_mur(float old_in, float new_in, float old_wall, float km) {
    return fmaf(km, new_in - old_wall, old_in);
}

// The update of FIELD_NODES nodes of one run (block `blk` of the block table) by T
// threads, FIELD_NODES / T nodes each (one, by some of them, where that is below one): old and new fields live in separate buffers and
// the guard values are recomputed from the neighbours' old data, so that one launch does
// the whole step.  It also zeroes the current accumulators of the next step (two sets), or of the one after it (three) and
// adds the exact discrete Poynting flux through the two accounting planes.
struct FieldSmem {
    // old E on nodes [i0-2, i0+N+1]; old B on half nodes [i0-2, i0+N], overwritten in place by
    // B^{n+1/2}; E^{n+1} on nodes [i0-1, i0+N]
    float ey[FIELD_NODES + 4], ez[FIELD_NODES + 4], by[FIELD_NODES + 3], bz[FIELD_NODES + 3];
    float ney[FIELD_NODES + 2], nez[FIELD_NODES + 2];
};

template <int T, bool PDL>
__device__ __forceinline__ void field_block(const FieldParams& P, unsigned phase, int blk, FieldSmem& S) {
    constexpr int N = FIELD_NODES, K = (N + T - 1) / T;
    constexpr bool EVEN = N % T == 0;  // else not every thread has a node in each of the K rounds
    const int tid = threadIdx.x;
    const int run = P.blk_run[blk];
    const RunDev& R = P.runs[run];
    if (!R.active) return;  // block-uniform
    const int i0 = P.blk_i0[blk];
    const int Nx = R.Nx, is = R.is, glen = R.glen;
    const int par = field_buf(R, phase), cur = current_set(R, phase, P.nsets);
    const float* const Fo[5] = {R.F[par][0], R.F[par][1], R.F[par][2], R.F[par][3], R.F[par][4]};
    float* const* Fn = R.F[1 - par];
    const unsigned long long* const Jacc[3] = {R.J[cur][0], R.J[cur][1], R.J[cur][2]};
    const int next = current_set(R, phase + P.nsets - 1, P.nsets);
    unsigned long long* const* Jnext = R.J[next];
    const float* inc = P.inc + 6 * run;
    const float c = P.c, hc = P.hc, fdt = P.fdt, fpi = R.fp_inv, fph = R.fp_inv * 4294967296.0f;
    pdl_wait<PDL>();

    // Every load of the block is issued here, before the first barrier: the old fields and the
    // transverse current of the stencil (J on node i0-1+q kept in the register of the thread that
    // updates E there), and Ex and Jx of the owned nodes.
    unsigned long long jy[K + 1], jz[K + 1], jx[K];
    float ex[K];
#pragma unroll
    for (int k = 0; k <= K; ++k) {
        const int q = tid + k * T;
        if ((k == K || !EVEN) && q >= N + 4) break;  // the 4 guard entries past the tile
        const int i = i0 - 2 + q + PADF;  // padded index, >= PADF - 2 >= 0
        const bool in = i < glen;         // the last block reaches past the array end
        S.ey[q] = in ? Fo[1][i] : 0.f;
        S.ez[q] = in ? Fo[2][i] : 0.f;
        if (q < N + 3) {
            S.by[q] = in ? Fo[3][i] : 0.f;
            S.bz[q] = in ? Fo[4][i] : 0.f;
        }
        // J on node i0-1+q for q < N+2 (one further than the old fields: index i+1)
        const bool jin = q < N + 2 && i + 1 < glen;
        jy[k] = jin ? Jacc[1][i + 1] : 0ull;
        jz[k] = jin ? Jacc[2][i + 1] : 0ull;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int q = tid + k * T, pi = i0 + q + PADF;
        const bool own = (EVEN || q < N) && i0 + q < Nx;
        jx[k] = own ? Jacc[0][pi] : 0ull;
        ex[k] = own ? Fo[0][pi] : 0.f;
    }
    __syncthreads();

    // B^{n+1/2} on half nodes j = i0-2+q, in place (entry q is read and written by one thread only)
#pragma unroll
    for (int k = 0; k <= K; ++k) {
        const int q = tid + k * T;
        if ((k == K || !EVEN) && q >= N + 3) break;
        float by = S.by[q], bz = S.bz[q];
        yee_b(by, bz, S.ey[q], S.ey[q + 1], S.ez[q], S.ez[q + 1], hc, i0 - 2 + q == is - 1, inc[0], inc[1]);
        S.by[q] = by;
        S.bz[q] = bz;
    }
    __syncthreads();

    // E^{n+1} on nodes i = i0-1+q (interior formula; Mur nodes below)
#pragma unroll
    for (int k = 0; k <= K; ++k) {
        const int q = tid + k * T;
        if ((k == K || !EVEN) && q >= N + 2) break;
        const int i = i0 - 1 + q;
        // node i: old E at sE[q+1], half nodes i-1, i at sB[q], sB[q+1]
        float ey = S.ey[q + 1], ez = S.ez[q + 1];
        yee_e(ey, ez, S.by[q], S.by[q + 1], S.bz[q], S.bz[q + 1], fix_to_float(jy[k], fpi, fph),
              fix_to_float(jz[k], fpi, fph), c, fdt, i == is, inc[2], inc[3]);
        const bool inner = i >= 1 && i <= Nx - 1;
        S.ney[q] = inner ? ey : 0.f;
        S.nez[q] = inner ? ez : 0.f;
    }
    __syncthreads();
    if (i0 == 0 || i0 + N >= Nx) {  // block-uniform: a wall (or the node before it) is in this block
        if (tid == 0) {
            const float km = (c - 1.f) / (c + 1.f);
            if (i0 - 1 <= 0 && 0 <= i0 + N) {
                const int q = 0 - (i0 - 1);
                // node 0: old at sE[q+1], node 1 old at sE[q+2], new node 1 at nE[q+1]
                S.ney[q] = yee_mur(S.ey[q + 2], S.ney[q + 1], S.ey[q + 1], km);
                S.nez[q] = yee_mur(S.ez[q + 2], S.nez[q + 1], S.ez[q + 1], km);
            }
            if (i0 - 1 <= Nx && Nx <= i0 + N) {
                const int q = Nx - (i0 - 1);
                S.ney[q] = yee_mur(S.ey[q], S.ney[q - 1], S.ey[q + 1], km);
                S.nez[q] = yee_mur(S.ez[q], S.nez[q - 1], S.ez[q + 1], km);
            }
        }
        __syncthreads();
    }

    // owned outputs: node / half node i = i0 + q
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int q = tid + k * T;  // node i: nE[q+1], sE[q+2]; half node i: sB[q+2]
        if (!EVEN && q >= N) break;
        const int i = i0 + q;
        const int pi = i + PADF;
        if (i <= Nx) {
            Fn[1][pi] = S.ney[q + 1];
            Fn[2][pi] = S.nez[q + 1];
        }
        if (i < Nx) {
            float by = S.by[q + 2], bz = S.bz[q + 2];
            yee_b(by, bz, S.ney[q + 1], S.ney[q + 2], S.nez[q + 1], S.nez[q + 2], hc, i == is - 1, inc[4], inc[5]);
            Fn[3][pi] = by;
            Fn[4][pi] = bz;
            Fn[0][pi] = fmaf(-fdt, fix_to_float(jx[k], fpi, fph), ex[k]);
        }
        // exact discrete Poynting flux through the accounting planes
        const int a = is + 1, b = Nx - 1;
        if (i == a) {
            const double ey = 0.5 * (static_cast<double>(S.ey[q + 2]) + S.ney[q + 1]);
            const double ez = 0.5 * (static_cast<double>(S.ez[q + 2]) + S.nez[q + 1]);
            R.tally[1] += P.dt * (ey * S.bz[q + 1] - ez * S.by[q + 1]);
        }
        if (i == b) {
            const double ey = 0.5 * (static_cast<double>(S.ey[q + 2]) + S.ney[q + 1]);
            const double ez = 0.5 * (static_cast<double>(S.ez[q + 2]) + S.nez[q + 1]);
            R.tally[2] += P.dt * (ey * S.bz[q + 2] - ez * S.by[q + 2]);
        }
    }
    // zero the accumulators of a later step: owned padded range of this block
    {
        const int lo = (i0 == 0) ? 0 : i0 + PADF;
        const int hi = (i0 + N > Nx) ? Nx + 2 * PADF + 1 : i0 + N + PADF;
        for (int pi = lo + tid; pi < hi; pi += T) {
            Jnext[0][pi] = 0ull;
            Jnext[1][pi] = 0ull;
            Jnext[2][pi] = 0ull;
        }
    }
}

}  // namespace picrr
