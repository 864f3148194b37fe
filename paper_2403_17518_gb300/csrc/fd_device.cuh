// Device helpers shared by the finite-difference step kernels (fd_kernels.cu,
// fd_tma.cu): stencil weights, tile types, packed two-lane FP32 arithmetic,
// the difference-form Laplacian, source injection, the sponge factor and
// receiver sampling.  Formulas: Section 2.1, Eq. 1 (see fd_kernels.cu).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include "fd_internal.h"

namespace dhfwi {

// 8th-order central second-difference weights for unit spacing (c0 is
// implied by c0 = -2 (c1 + c2 + c3 + c4)).
#define FD_C1 (8.0f / 5.0f)
#define FD_C2 (-1.0f / 5.0f)
#define FD_C3 (8.0f / 315.0f)
#define FD_C4 (-1.0f / 560.0f)

typedef float STile[SROWS][SROW];
typedef float CTile[TZ][TX];

// ---------------------------------------------------------------------------
// Packed two-lane FP32 arithmetic (sm_100+ add/sub/mul/fma .f32x2): lane 0 is
// the low word (float2.x).  Each lane is rounded exactly like the scalar op.
// ---------------------------------------------------------------------------
typedef unsigned long long f2;
__device__ __forceinline__ f2 pk(float2 a) { return *reinterpret_cast<f2 *>(&a); }
__device__ __forceinline__ float2 upk(f2 a) { return *reinterpret_cast<float2 *>(&a); }
__device__ __forceinline__ f2 pk2(float lo, float hi) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

// Difference-form D u for the two cells (row lzr, columns lxp, lxp+1) of a
// thread, both lanes at once.  zc holds the two columns for rows lzr-4 ..
// lzr+4 (index 4 = the cells).
// rp: the row segment of the two cells, columns x-4 .. x+5 as five float2
// (the cells are x, x+1); zc: the two columns for rows -4 .. +4.
__device__ __forceinline__ f2 lap8x2_seg(const float2 *rp, const float2 *zc) {
    const float2 r0 = rp[0], r1 = rp[1], r2 = rp[2], r3 = rp[3], r4 = rp[4];
    // r0=(x-4,x-3) r1=(x-2,x-1) r2=(x,x+1) r3=(x+2,x+3) r4=(x+4,x+5)
    const f2 u = pk(r2);
    const f2 m4 = pk(r0), p4 = pk(r4);
    const f2 m3 = pk2(r0.y, r1.x), p3 = pk2(r3.y, r4.x);
    const f2 m2 = pk(r1), p2 = pk(r3);
    const f2 m1 = pk2(r1.y, r2.x), p1 = pk2(r2.y, r3.x);
    const f2 c1 = pk2(FD_C1, FD_C1), c2 = pk2(FD_C2, FD_C2), c3 = pk2(FD_C3, FD_C3), c4 = pk2(FD_C4, FD_C4);
    f2 a = mul2(c4, add2(add2(sub2(p4, u), sub2(m4, u)), add2(sub2(pk(zc[8]), u), sub2(pk(zc[0]), u))));
    a = fma2(c3, add2(add2(sub2(p3, u), sub2(m3, u)), add2(sub2(pk(zc[7]), u), sub2(pk(zc[1]), u))), a);
    a = fma2(c2, add2(add2(sub2(p2, u), sub2(m2, u)), add2(sub2(pk(zc[6]), u), sub2(pk(zc[2]), u))), a);
    a = fma2(c1, add2(add2(sub2(p1, u), sub2(m1, u)), add2(sub2(pk(zc[5]), u), sub2(pk(zc[3]), u))), a);
    return a;
}
__device__ __forceinline__ f2 lap8x2(const STile &s, const float2 *zc, int lzr, int lxp) {
    // Row segment: columns lxp .. lxp+9 (the cells sit at lxp+4, lxp+5).
    return lap8x2_seg(reinterpret_cast<const float2 *>(&s[lzr + HALO][lxp]), zc);
}

// ---------------------------------------------------------------------------
// Four adjacent columns of one row (16-byte shared and global accesses).
// ---------------------------------------------------------------------------
struct q4 {
    f2 lo, hi;
};
__device__ __forceinline__ q4 ld4(const float *p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p);
    return q4{v.x, v.y};
}
__device__ __forceinline__ void st4(float *p, q4 v) { *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(v.lo, v.hi); }
__device__ __forceinline__ q4 add4(q4 a, q4 b) { return q4{add2(a.lo, b.lo), add2(a.hi, b.hi)}; }
__device__ __forceinline__ q4 mul4(q4 a, q4 b) { return q4{mul2(a.lo, b.lo), mul2(a.hi, b.hi)}; }
__device__ __forceinline__ q4 fma4(q4 a, q4 b, q4 c) { return q4{fma2(a.lo, b.lo, c.lo), fma2(a.hi, b.hi, c.hi)}; }

// One ring of the difference-form D u (see lap8x2_seg): right, left, lower
// and upper neighbours of two cells.
__device__ __forceinline__ f2 lap_ring(f2 p, f2 m, f2 zp, f2 zm, f2 u) {
    return add2(add2(sub2(p, u), sub2(m, u)), add2(sub2(zp, u), sub2(zm, u)));
}

// D u down a column of quads in a shared-memory tile of row pitch P, with
// lap8x2_seg's operations in its order.  p points at the quad, four rows above
// the first row; rows are taken in order, each row of the column read once.
template <int P>
struct LapColumn {
    const float *p;
    q4 c[9];  // the rows around the current one, as a ring
    __device__ __forceinline__ explicit LapColumn(const float *p_) : p(p_) {
#pragma unroll
        for (int r = 0; r < 8; r++) c[r] = ld4(p + r * P);
    }
    // Row rr (a compile-time constant after unrolling): D u and u itself.
    __device__ __forceinline__ q4 row(int rr, q4 &u) {
        c[(rr + 8) % 9] = ld4(p + (rr + 8) * P);
        auto z = [&](int k) { return c[(rr + 4 + k) % 9]; };
        const float *r = p + (rr + 4) * P;
        const q4 L = ld4(r - 4), R = ld4(r + 4), C = z(0);
        u = C;
        const float2 l0 = upk(L.lo), l1 = upk(L.hi), c0 = upk(C.lo), c1 = upk(C.hi), r0 = upk(R.lo), r1 = upk(R.hi);
        // Pairs that start at odd columns: x-3, x-1, x+1, x+3, x+5.
        const f2 b0 = pk2(l0.y, l1.x), b1 = pk2(l1.y, c0.x), b2 = pk2(c0.y, c1.x), b3 = pk2(c1.y, r0.x),
                 b4 = pk2(r0.y, r1.x);
        const f2 w1 = pk2(FD_C1, FD_C1), w2 = pk2(FD_C2, FD_C2), w3 = pk2(FD_C3, FD_C3), w4 = pk2(FD_C4, FD_C4);
        f2 a = mul2(w4, lap_ring(R.lo, L.lo, z(4).lo, z(-4).lo, C.lo));
        a = fma2(w3, lap_ring(b3, b0, z(3).lo, z(-3).lo, C.lo), a);
        a = fma2(w2, lap_ring(C.hi, L.hi, z(2).lo, z(-2).lo, C.lo), a);
        a = fma2(w1, lap_ring(b2, b1, z(1).lo, z(-1).lo, C.lo), a);
        f2 e = mul2(w4, lap_ring(R.hi, L.hi, z(4).hi, z(-4).hi, C.hi));
        e = fma2(w3, lap_ring(b4, b1, z(3).hi, z(-3).hi, C.hi), e);
        e = fma2(w2, lap_ring(R.lo, C.lo, z(2).hi, z(-2).hi, C.hi), e);
        e = fma2(w1, lap_ring(b3, b2, z(1).hi, z(-1).hi, C.hi), e);
        return q4{a, e};
    }
};

// Source injection into lane 0 / 1 of a when the cell is the source node.
__device__ __forceinline__ f2 inject(f2 a, int i, int j, int sz, int sx, float q) {
    if (i == sz && (j == sx || j + 1 == sx)) {
        float2 v = upk(a);
        if (j == sx) v.x += q;
        else v.y += q;
        a = pk(v);
    }
    return a;
}

// Cerjan sponge factor along one axis: exp(-(0.015 (nb - d))^2), d = cells
// from the outer edge; 1 inside.
__device__ __forceinline__ float sponge1(int i, int N, int nb) {
    const int d = min(i, N - 1 - i);
    const int p = nb - d;
    return p > 0 ? expf(-2.25e-4f * (float)(p * p)) : 1.0f;
}

template <int NT>
__device__ __forceinline__ void sample_receivers(const STile &so, const Tile &t, const Tile &tn,
                                                 const TileRec *__restrict__ recs, const ShotDesc &sd,
                                                 float *__restrict__ d, int n) {
    const int tid = threadIdx.x + threadIdx.y * 32;
    for (int e = t.rec_begin + tid; e < tn.rec_begin; e += NT) {
        const TileRec tr = recs[e];
        d[sd.doff + (long long)n * sd.nrec + tr.r] = so[tr.cell / TX + HALO][tr.cell % TX + HALO];
    }
}

// Model arrays are stored as 4 copies, copy r shifted left by r columns, so
// the model row of a window starting at model column x0 is 16-byte aligned in
// copy (x0 & 3) at column (x0 & ~3).
__device__ __forceinline__ const float *model_base(const float *arr, const StepCommon &c, int x0) {
    return arr + (long long)(x0 & 3) * c.mstride + (x0 & ~3);
}

template <typename T>
__device__ __forceinline__ T &sm2(float *p) { return *reinterpret_cast<T *>(p); }

// Receiver injection of one adjoint step into a TZ x TX tile: inj[cell] =
// the sum of the data sample rk[r] over the tile's receivers at that cell,
// zero elsewhere.  A tile's receiver entries are sorted by cell, then by
// receiver, so duplicates are summed in a fixed order by the thread that
// owns the first entry of their cell (deterministic, no atomics).  Ends
// with a barrier.
__device__ __forceinline__ float receiver_sum(const TileRec *__restrict__ recs, int e, int re,
                                              const float *__restrict__ rk) {
    const int cell = recs[e].cell;
    float s = rk[recs[e].r];
    for (int f = e + 1; f < re && recs[f].cell == cell; f++) s += rk[recs[f].r];
    return s;
}
template <int NT>
__device__ __forceinline__ void build_injection(CTile &inj, const TileRec *__restrict__ recs, int rb, int re,
                                                const float *__restrict__ rk, int tid) {
    for (int e = tid; e < TZ * TX; e += NT) (&inj[0][0])[e] = 0.f;
    __syncthreads();
    for (int e = rb + tid; e < re; e += NT)
        if (e == rb || recs[e - 1].cell != recs[e].cell) {
            const int cell = recs[e].cell;
            inj[cell / TX][cell % TX] = receiver_sum(recs, e, re, rk);
        }
    __syncthreads();
}

// Lane 1 (column j+1) cleared when it lies past the window (odd widths), so
// the padding columns of a field pool stay zero: tiles staged straight from
// a pool read them as the zero boundary.
__device__ __forceinline__ f2 keep_lo(f2 v, bool hi) { return hi ? v : (v & 0xffffffffull); }

}  // namespace dhfwi
