// Two-step (time-blocked) forward, adjoint and Born kernels for sm_103a: one
// launch advances every active tile by two steps of the recurrence of Section 2.1
// (Eq. 1, summed form; see fd_kernels.cu), so u and D cross HBM once per two
// updates.
//
// Per 64 x 64 tile the TMA stages u^n with an 8-cell halo and D^n with a
// 4-cell ring.  Step n is computed on the tile and its ring, giving
// u^{n+1} in shared memory (zero outside the window: the Dirichlet boundary);
// step n+1 is then computed on the core from it.  The ring cells are
// recomputed by each tile that needs them (1024 per 4096, the corners, which
// no stencil reaches, left out), so tiles never exchange data within the
// launch; since they read D^n on their neighbours' cells, D^{n+2} goes to a
// second pool.  Every cell goes through the same floating-point operations in
// the same order as in the one-step kernels, so the results are bit-identical.
//
// Work split: an item is 4 columns x 4 rows.  The 256 items of the core
// belong to warps 0-7, the 32 left and right ring items to warp 8, the 32 top
// and bottom ones to warp 9: ten full warps in step n, and a core thread
// advances the same 16 cells in both steps, so D^{n+1} only passes through the
// thread's own 64 bytes of shared memory.  16-byte accesses take 1.9 shared
// loads per update where two columns per thread took 5.7.  kappa, shared by
// all shots and L2-resident, is copied by each thread into slots of its own a
// tile ahead (cp.async): no thread waits on a global load between the barriers.
// What bounds it: latency at 20 warps per SM.  Forward, 64 shots of 400 x 1200,
// per launch: 64.4 us (two columns x 9 rows per thread, sponge factors and
// bounds tests computed per row) -> 58.8 (items, kappa and sponge factors loaded
// where they are used) -> 48.5 (both copied a tile ahead) -> 47.5 (kappa awaited
// only where it is used, after the first Laplacian; storing a^n: 58 -> 54 us).
//
// Sponge: the factor is separable and depends on the distances to the padded
// domain's edges only, so the plan holds it per row and per slot's column
// (zero outside the domain, which also masks the cells out there); the tile's
// 72 + 72 factors are copied a tile ahead, and a tile that the sponge reaches
// needs no bounds tests.
//
// Sources: injected at both steps (q^n, q^{n+1}), also on ring cells.
// Receivers: sample n from u^{n+1} in shared memory, sample n+1 from the
// pool after the tile's stores.  Checkpoints (u^n, D^n) at even n, history or
// segment stores of a^n and a^{n+1}.  Tiles of a shot whose record ends at n+1
// take step n only.
#include <cuda.h>
#include <cuda_runtime.h>

#include "fd_tma.cuh"

namespace dhfwi {
namespace {

constexpr int E = TX + 2 * HALO;     // 72: core + ring
constexpr int U2R = TZ + 2 * HALO2;  // 80 rows of the u^n box
static_assert(TX == TZ && TX == 64 && HALO == 4, "the item layout below");
// Row pitches with 4 rows off a multiple of the 32 banks, so that the ring
// items of one column of quads spread over them (u: box of 84 columns).
constexpr int VP = 76;
struct Pair2Stage {
    float u[U2R][U2PITCH];  // u^n: rows z0-8 .., cols x0-8 ..
    float d[E][E];          // D^n: rows z0-4 .., cols x0-4 ..
};
constexpr unsigned kPair2StageBytes = sizeof(float) * (U2R * U2PITCH + E * E);
static_assert(sizeof(Pair2Stage) == kPair2StageBytes, "stage layout");
static_assert(U2R * U2PITCH * 4 % 128 == 0 && E * E * 4 % 128 == 0, "TMA destinations stay 128-byte aligned");
typedef float VTile[E][VP];  // u^{n+1}: rows z0-4 .., cols x0-4 ..
// The stage's barrier and the descriptors of this tile, the next one (whose
// loads the leader issues in the middle of this one) and the one after.
struct PairTail {
    unsigned long long bar[2];
    TileInfo desc[3];
};
static_assert(sizeof(PairTail) % 16 == 0, "tail layout");
// Per-thread 16-byte slots: kappa of the thread's item (row rr at k[rr]),
// which the thread copies itself (cp.async) for the next tile once it is done
// with this one's, so that it needs no barrier; and D^{n+1} of the core threads'
// cells between the steps.
struct ItemSlots {
    float4 k[4][320], d[4][256];
};
// Two-step Born: kappa and d kappa; the core's D_p^{n+1} stays in registers.
struct BornSlots {
    float4 k[4][320], dk[4][320];
};
// Sponge factors of the tile's rows and columns, ring included; this tile's
// and the next one's alternate.
struct TileEdge {
    float wz[E], wx[E];
};
template <class Slots>
constexpr size_t pair_smem() {
    return sizeof(Pair2Stage) + sizeof(VTile) + sizeof(Slots) + 2 * sizeof(TileEdge) + sizeof(PairTail);
}
constexpr size_t kPair2Smem = pair_smem<ItemSlots>(), kBorn2Smem = pair_smem<BornSlots>();
// The two-step adjoint's list of its next tile's data injection (grown
// region, step k): offset of the cell in the staged D_nu (-1: a further
// receiver of the cell before, already summed), kappa there, summed data.
struct InjEntry {
    int off;
    float kap, sum;
};
struct InjBuf {
    int n, pad[3];
    InjEntry e[kInjCap];
};
constexpr size_t kAdj2Smem = kPair2Smem + sizeof(InjBuf);
static_assert(kPair2Smem % 16 == 0, "injection list alignment");

constexpr int NT2 = 320, NCORE = 256, R4 = 4;
constexpr int LEADER2 = 288;  // first thread of warp 9, which is free during step n+1

// Core-relative column and first row of a thread's item (4 columns x R rows):
// the core's items, then the left and right ring's alternately, then the top
// and bottom ring's.
template <int R>
__device__ __forceinline__ void item_of(int tid, int &lx, int &lz) {
    constexpr int NC = 16 * (TZ / R), NS = 2 * (TZ / R);
    if (tid < NC) {
        lx = 4 * (tid & 15);
        lz = R * (tid >> 4);
    } else if (tid < NC + NS) {
        const int i = tid - NC;
        lx = (i & 1) ? TX : -HALO;
        lz = R * (i >> 1);
    } else {
        const int i = tid - NC - NS, z = i >> 4;  // z: HALO / R blocks above, then below
        lx = 4 * (i & 15);
        lz = z < HALO / R ? R * z - HALO : TZ + R * z - HALO;
    }
}

// The source cell of a thread's item, as 4 * row + column, or -1.
template <int R>
__device__ __forceinline__ int item_source(const TileInfo &T, int lx, int lz) {
    const unsigned x = T.sx - (T.x0 + lx), z = T.sz - (T.z0 + lz);
    return x < 4u && z < (unsigned)R ? (int)(4 * z + x) : -1;
}
// Sponge factors of the item's row rr.
__device__ __forceinline__ q4 row_w(const TileEdge &We, int lx, int lz, int rr) {
    const float z = We.wz[lz + rr + HALO];
    const q4 x = ld4(&We.wx[lx + HALO]);
    return q4{mul2(pk2(z, z), x.lo), mul2(pk2(z, z), x.hi)};
}
// This thread's cells of a model array (kappa, d kappa; L2-resident) into its
// slots.  Rows and quads outside the padded domain, whose sponge factor is
// zero, take some cell's inside it.
template <int R, int NT>
__device__ __forceinline__ void copy_item(float4 (*slots)[NT], const float *model, const StepCommon &c,
                                          const TileInfo &T, int tid) {
    int lx, lz;
    item_of<R>(tid, lx, lz);
    const float *m = model + (long long)T.mc * c.mstride + min(max(T.mx + lx, 0), c.pf - 4);
#pragma unroll
    for (int rr = 0; rr < R; rr++)
        cp_async16(&slots[rr][tid], m + min(max(T.z0 + lz + rr, 0), c.NZ - 1) * c.pf);
}
// A tile's sponge factors, copied by one warp.
__device__ __forceinline__ void copy_edge(TileEdge &We, const StepCommon &c, const TileInfo &T, int lane) {
    if (lane < E / 4) {
        cp_async16(&We.wz[4 * lane], c.wz + T.z0 + 4 * lane);
        cp_async16(&We.wx[4 * lane], c.wx + (long long)T.slot * (T.pitch + 2 * HALO) + T.x0 + 4 * lane);
    }
}
__device__ __forceinline__ void add_source(q4 &a, int scol, float q) {
    float2 l = upk(a.lo), h = upk(a.hi);
    if (scol == 0) l.x += q;
    if (scol == 1) l.y += q;
    if (scol == 2) h.x += q;
    if (scol == 3) h.y += q;
    a = q4{pk(l), pk(h)};
}

// mid(): called by every thread after the barrier that ends step n (the
// stage is no longer read): the leader refills the stage.
// STORE: what else a launch stores (nothing, a^n and a^{n+1}, or the
// checkpoint u^n, D^n).
enum { ST_NONE = 0, ST_A = 1, ST_CK = 2 };
template <int STORE, bool FULL, class MidFn>
__device__ __forceinline__ void pair_tile(const FwdArgs &A, const Pair2Stage &S, VTile &V, ItemSlots &I, const TileEdge &We,
                                          const TileInfo &T, int tid, bool two, MidFn mid) {
    int lx, lz;
    item_of<R4>(tid, lx, lz);
    const bool core = tid < NCORE;
    const int n = A.n, pitch = T.pitch;
    const int j = T.x0 + lx, i0 = T.z0 + lz;
    const int nrow = FULL ? R4 : A.c.NZ - i0;
    const bool ok = core && (FULL || j < T.nxw);
    const long long cbase = T.foff + (long long)i0 * pitch + j;
    const int src = FULL ? -1 : item_source<R4>(T, lx, lz);

    // ---- step n on the item ------------------------------------------------
    {
        LapColumn<U2PITCH> col(&S.u[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            q4 u;
            q4 a = col.row(rr, u);
            if (rr == 0) cp_async_wait<0>();
            const q4 dv = ld4(&S.d[lz + rr + HALO][lx + HALO]);
            const q4 kv = ld4(&I.k[rr][tid].x);
            q4 un, dn;
            if constexpr (FULL) {
                dn = fma4(kv, a, dv);
                un = add4(u, dn);
            } else {
                if (rr == src >> 2) add_source(a, src & 3, A.c.wav[T.wav_off + n]);
                const q4 w = row_w(We, lx, lz, rr);
                dn = mul4(w, fma4(kv, a, dv));
                un = fma4(w, u, dn);
            }
            st4(&V[lz + rr + HALO][lx + HALO], un);
            if (core) st4(&I.d[rr][tid].x, dn);
            if (ok && rr < nrow) {
                const long long c = cbase + (long long)rr * pitch;
                if constexpr (STORE == ST_CK) {
                    st4(A.ck_u + c, u);
                    st4(A.ck_d + c, dv);
                }
                if constexpr (STORE == ST_A) st4(A.a_out + c, a);
            }
        }
    }
    __syncthreads();  // u^{n+1} complete; the stage is no longer read
    mid();

    // Receivers: sample n is u^{n+1} (the ring warps, free from here on).
    if (A.d && !core) {
        for (int e = T.rec_begin + tid - NCORE; e < T.rec_end; e += NT2 - NCORE) {
            const TileRec tr = A.c.recs[e];
            A.d[T.doff + (long long)n * T.nrec + tr.r] = V[tr.cell / TX + HALO][tr.cell % TX + HALO];
        }
    }

    // ---- step n+1 on the core ----------------------------------------------
    if (!two) {  // the record ends at n+1: store u^{n+1}, D^{n+1}
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            if (ok && rr < nrow) {
                const long long c = cbase + (long long)rr * pitch;
                st4(A.un + c, ld4(&V[lz + rr + HALO][lx + HALO]));
                st4(A.dd_out + c, ld4(&I.d[rr][tid].x));
            }
        }
        return;
    }
    if (ok) {
        LapColumn<VP> col(&V[lz][lx + HALO]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            q4 u;
            q4 a = col.row(rr, u);
            const q4 kv = ld4(&I.k[rr][tid].x), dn = ld4(&I.d[rr][tid].x);
            q4 d2, un;
            if constexpr (FULL) {
                d2 = fma4(kv, a, dn);
                un = add4(u, d2);
            } else {
                if (rr == src >> 2) add_source(a, src & 3, A.c.wav[T.wav_off + n + 1]);
                const q4 w = row_w(We, lx, lz, rr);
                d2 = mul4(w, fma4(kv, a, dn));
                un = fma4(w, u, d2);
            }
            if (rr < nrow) {
                const long long c = cbase + (long long)rr * pitch;
                st4(A.dd_out + c, d2);
                st4(A.un + c, un);
                if constexpr (STORE == ST_A) st4(A.a_out2 + c, a);
            }
        }
    }
    // Receivers: sample n+1 is u^{n+2}, read back from the pool.
    if (A.d && T.rec_end > T.rec_begin) sample_from_pool<NT2>(A.c, T, A.un, A.d, n + 1);
}

// What the tile loop itself uses of a kernel's shared memory.
struct PairLoopSmem {
    const void *stage;
    TileEdge *We;
    PairTail *tail;
};
// Shared memory of a two-step kernel of one field.
template <class Slots>
struct PairSmem {
    Pair2Stage &S;
    VTile &V;
    Slots &I;
    TileEdge *We;
    PairTail *tail;
    __device__ __forceinline__ explicit PairSmem(unsigned char *m)
        : S(*reinterpret_cast<Pair2Stage *>(m)), V(*reinterpret_cast<VTile *>(m + sizeof(Pair2Stage))),
          I(*reinterpret_cast<Slots *>(m + sizeof(Pair2Stage) + sizeof(VTile))),
          We(reinterpret_cast<TileEdge *>(m + sizeof(Pair2Stage) + sizeof(VTile) + sizeof(Slots))),
          tail(reinterpret_cast<PairTail *>(We + 2)) {}
    __device__ __forceinline__ PairLoopSmem loop() const { return {&S, We, tail}; }
};

// Tile loop: one stage, refilled in the middle of a tile so that the next
// tile's loads overlap step n+1; the barrier that opens a tile also certifies
// that every thread is done with the tile before (V, and the descriptor slot,
// which alternates).  Waits bounded as in run_tiles.
//   issue(T, bar): the leader's tensor loads of a tile's stage;
//   fill(T): every thread's copies of a tile's model values into its slots
//     (body awaits them with cp_async_wait<0>() before their first use: no
//     other thread reads them, so their latency overlaps the opening barrier
//     and the first Laplacian);
//   begin(t): before the first tile t, by every thread, no barrier inside;
//   open(): once a tile's stage has landed (may synchronise the CTA);
//   body(T, We, mid): the tile, calling mid() after the barrier that ends step
//     n (the stage is no longer read then: the leader refills it);
//   close(t): after the tile, t the next one.
// BYTES: the stage's, LEADER: the first thread of the warp that refills it.
template <unsigned BYTES, int LEADER, class IssueFn, class FillFn, class BeginFn, class OpenFn, class BodyFn,
          class CloseFn>
__device__ __forceinline__ void run_pairs(const StepCommon &c, int ntiles, const PairLoopSmem &P, int tid,
                                          IssueFn issue, FillFn fill, BeginFn begin, OpenFn open, BodyFn body,
                                          CloseFn close) {
    const bool leader = tid == LEADER;
    const unsigned bar = smem_u32(&P.tail->bar[0]);
    const int b = blockIdx.x, g = gridDim.x;
    if (smem_u32(P.stage) & 127u) {
        if (leader) atomicExch(c.tflag, 2u);
        return;
    }
    if (leader) {
        mbar_init(bar, 1);
        fence_mbar_init();
        copy_desc(&P.tail->desc[0], &c.infos[b]);
        if (b + g < ntiles) copy_desc(&P.tail->desc[1], &c.infos[b + g]);
        cp_async_wait_all();
    }
    griddep_wait();
    griddep_launch_dependents();
    auto refill = [&](const TileInfo &N) {
        fence_proxy_async();
        mbar_expect_tx(bar, BYTES);
        issue(N, bar);
    };
    if (leader) refill(P.tail->desc[0]);
    begin(b);
    __syncthreads();
    if (tid >= LEADER) copy_edge(P.We[0], c, P.tail->desc[0], tid - LEADER);
    cp_async_commit();
    fill(P.tail->desc[0]);
    cp_async_commit();
    unsigned phase = 0;
    int slot = 0, next = 1;
    for (int tix = b; tix < ntiles; tix += g) {
        const bool landed = mbar_wait(bar, phase);
        phase ^= 1u;
        cp_async_wait<1>();  // all but the thread's own slots, which it waits for before it reads them
        if (__syncthreads_or(!landed)) {
            cp_async_wait<0>();
            if (leader) {
                mbar_wait(bar, phase ^ 1u);  // copies in flight: a second bounded wait before leaving
                atomicExch(c.tflag, 1u);
            }
            return;
        }
        open();
        const bool more = tix + g < ntiles;
        auto mid = [&]() {  // after a barrier: every thread is done with the stage
            if (tid < LEADER || !more) return;
            if (leader) {
                refill(P.tail->desc[next]);
                if (tix + 2 * g < ntiles) copy_desc(&P.tail->desc[3 - slot - next], &c.infos[tix + 2 * g]);
            }
            copy_edge(P.We[phase], c, P.tail->desc[next], tid - LEADER);
        };
        body(P.tail->desc[slot], P.We[phase ^ 1u], mid);
        cp_async_commit();  // (the copies of mid())
        if (more) {
            fill(P.tail->desc[next]);
            close(tix + g);
        }
        cp_async_commit();
        const int after = 3 - slot - next;
        slot = next;
        next = after;
    }
}

template <int STORE>
__global__ void __launch_bounds__(NT2, 2) fwd_pair_kernel(FwdArgs A, const __grid_constant__ TileMaps M, int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PairSmem<ItemSlots> P(smem_raw);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_pairs<kPair2StageBytes, LEADER2>(
        A.c, ntiles, P.loop(), tid,
        [&](const TileInfo &N, unsigned bar) {
            tma_load_3d(smem_u32(&P.S.u), &M.m[0], N.x0 - HALO2, N.z0 - HALO2, N.slot, bar);
            tma_load_3d(smem_u32(&P.S.d), &M.m[1], N.x0 - HALO, N.z0 - HALO, N.slot, bar);
        },
        [&](const TileInfo &N) { copy_item<R4>(P.I.k, A.c.kap, A.c, N, tid); },
        [](int) {}, []() {},
        [&](const TileInfo &T, const TileEdge &We, auto mid) {
            const bool two = T.nt > A.n + 1;
            if (T.flags & TI_FULL2) pair_tile<STORE, true>(A, P.S, P.V, P.I, We, T, tid, two, mid);
            else pair_tile<STORE, false>(A, P.S, P.V, P.I, We, T, tid, two, mid);
        },
        [](int) {});
}

// ---------------------------------------------------------------------------
// Two-step Born from a^n (see born_hist_tma_kernel): the scattered field p
// advances by the steps n and n+1 with the background terms a^n and a^{n+1} of
// a stored forward pass.  The layout
// of fwd_pair_kernel, with d kappa in slots beside kappa; a^n, read once per
// step, is prefetched into L2 a tile ahead and loaded a row ahead.
// ---------------------------------------------------------------------------
template <bool FULL, class MidFn>
__device__ __forceinline__ void born_pair_tile(const BornArgs &A, const PairSmem<BornSlots> &P, const TileEdge &We,
                                               const TileInfo &T, int tid, bool two, MidFn mid) {
    int lx, lz;
    item_of<R4>(tid, lx, lz);
    const bool core = tid < NCORE;
    const int n = A.n, pitch = T.pitch, NZ = A.c.NZ;
    const int j = T.x0 + lx, i0 = T.z0 + lz;
    const int nrow = FULL ? R4 : NZ - i0;
    const bool ok = core && (FULL || j < T.nxw);
    const long long cbase = T.foff + (long long)i0 * pitch + j;
    // a outside the window reads as zero (its padding columns may hold anything).
    const bool in_x = FULL || (j >= 0 && j < T.nxw);
    auto load_a = [&](const float *a, int rr) {
        if (FULL) return ld4(a + cbase + (long long)rr * pitch);
        q4 v{0ull, 0ull};
        if (in_x && (unsigned)(i0 + rr) < (unsigned)NZ) {
            v = ld4(a + cbase + (long long)rr * pitch);
            const int w = T.nxw - j;  // columns of the quad inside the window
            if (w < 4) v = q4{w < 2 ? keep_lo(v.lo, false) : v.lo, w < 3 ? 0ull : keep_lo(v.hi, false)};
        }
        return v;
    };

    q4 dn[R4];

    // ---- step n on the item ------------------------------------------------
    {
        q4 an = load_a(A.a, 0);
        LapColumn<U2PITCH> col(&P.S.u[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            const q4 a0 = an;
            if (rr + 1 < R4) an = load_a(A.a, rr + 1);
            q4 p;
            const q4 ap = col.row(rr, p);
            if (rr == 0) cp_async_wait<0>();
            const q4 dv = ld4(&P.S.d[lz + rr + HALO][lx + HALO]);
            const q4 kv = ld4(&P.I.k[rr][tid].x), dkv = ld4(&P.I.dk[rr][tid].x);
            const q4 t = fma4(dkv, a0, fma4(kv, ap, dv));
            q4 pn;
            if constexpr (FULL) {
                dn[rr] = t;
                pn = add4(p, dn[rr]);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                dn[rr] = mul4(w, t);
                pn = fma4(w, p, dn[rr]);
            }
            st4(&P.V[lz + rr + HALO][lx + HALO], pn);
        }
    }
    __syncthreads();  // p^{n+1} complete; the stage is no longer read
    mid();

    // Receivers: sample n is p^{n+1} (the ring warps, free from here on).
    if (!core) {
        for (int e = T.rec_begin + tid - NCORE; e < T.rec_end; e += NT2 - NCORE) {
            const TileRec tr = A.c.recs[e];
            A.d[T.doff + (long long)n * T.nrec + tr.r] = P.V[tr.cell / TX + HALO][tr.cell % TX + HALO];
        }
    }
    if (!two) return;  // the record ends at n+1: the state is not needed any more

    // ---- step n+1 on the core ----------------------------------------------
    if (ok) {
        q4 an = load_a(A.a2, 0);
        LapColumn<VP> col(&P.V[lz][lx + HALO]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            const q4 a0 = an;
            if (rr + 1 < R4) an = load_a(A.a2, rr + 1);
            q4 p;
            const q4 ap = col.row(rr, p);
            const q4 kv = ld4(&P.I.k[rr][tid].x), dkv = ld4(&P.I.dk[rr][tid].x);
            const q4 t = fma4(dkv, a0, fma4(kv, ap, dn[rr]));
            q4 d2, pn;
            if constexpr (FULL) {
                d2 = t;
                pn = add4(p, d2);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                d2 = mul4(w, t);
                pn = fma4(w, p, d2);
            }
            if (rr < nrow) {
                const long long c = cbase + (long long)rr * pitch;
                st4(A.dp_out + c, d2);
                st4(A.pn + c, pn);
            }
        }
    }
    // Receivers: sample n+1 is p^{n+2}, read back from the pool.
    if (T.rec_end > T.rec_begin) sample_from_pool<NT2>(A.c, T, A.pn, A.d, n + 1);
}

__global__ void __launch_bounds__(NT2, 2) born_pair_kernel(BornArgs A, const __grid_constant__ TileMaps M, int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PairSmem<BornSlots> P(smem_raw);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_pairs<kPair2StageBytes, LEADER2>(
        A.c, ntiles, P.loop(), tid,
        [&](const TileInfo &N, unsigned bar) {
            tma_load_3d(smem_u32(&P.S.u), &M.m[0], N.x0 - HALO2, N.z0 - HALO2, N.slot, bar);
            tma_load_3d(smem_u32(&P.S.d), &M.m[1], N.x0 - HALO, N.z0 - HALO, N.slot, bar);
            tma_prefetch_l2_3d(&M.m[2], N.x0, N.z0, N.slot);
            tma_prefetch_l2_3d(&M.m[3], N.x0, N.z0, N.slot);
        },
        [&](const TileInfo &N) {
            copy_item<R4>(P.I.k, A.c.kap, A.c, N, tid);
            copy_item<R4>(P.I.dk, A.dkap, A.c, N, tid);
        },
        [](int) {}, []() {},
        [&](const TileInfo &T, const TileEdge &We, auto mid) {
            const bool two = T.nt > A.n + 1;
            if (T.flags & TI_INTERIOR2) born_pair_tile<true>(A, P, We, T, tid, two, mid);
            else born_pair_tile<false>(A, P, We, T, tid, two, mid);
        },
        [](int) {});
}

// ---------------------------------------------------------------------------
// Two-step Born, both fields (see born_tma_kernel): u0 and p advance by the
// steps n and n+1 in one launch, so each field crosses HBM once per two steps
// (16 bytes per cell and step of both, where the one-step kernel moves 32) and
// a^n stays in registers between the two updates of a cell.  Both fields' stages
// fill most of the shared memory, so one CTA of 20 warps takes a tile: items of
// 4 x 2 cells, 512 of the core and 128 of the ring.  Bound by shared-memory
// reads (53 % of the wavefronts) and latency at 20 warps per SM.  64 shots of
// 400 x 1200, 3983 steps: 272 ms (one step per launch, DRAM 64 % busy) -> 215 ms.
// A forward pair launch that stores a^n and a scattered-field one that reads it
// (24 bytes) took 270 ms.
// ---------------------------------------------------------------------------
constexpr int RJ = 2, NTJ = 640, NCOREJ = 512, LEADERJ = 608;
struct JointStage {
    float u[U2R][U2PITCH], p[U2R][U2PITCH];
    float du[E][E], dp[E][E];
};
constexpr unsigned kJointStageBytes = sizeof(JointStage);
struct JointSmem {
    JointStage S;
    VTile Vu, Vp;
    float4 k[RJ][NTJ], dk[RJ][NTJ], du[RJ][NCOREJ], dp[RJ][NCOREJ];  // per-thread slots, see ItemSlots
    TileEdge We[2];
    PairTail tail;
};
static_assert(sizeof(JointStage) == 8 * (U2R * U2PITCH + E * E) && sizeof(JointSmem) % 16 == 0, "stage layout");

template <bool FULL, class MidFn>
__device__ __forceinline__ void joint_tile(const BornArgs &A, JointSmem &P, const TileEdge &We, const TileInfo &T,
                                           int tid, bool two, MidFn mid) {
    int lx, lz;
    item_of<RJ>(tid, lx, lz);
    const bool core = tid < NCOREJ;
    const int n = A.n, pitch = T.pitch;
    const int j = T.x0 + lx, i0 = T.z0 + lz;
    const int nrow = FULL ? RJ : A.c.NZ - i0;
    const bool ok = core && (FULL || j < T.nxw);
    const int src = FULL ? -1 : item_source<RJ>(T, lx, lz);
    q4 a0[RJ];

    // ---- step n on the item: the background, then the scattered field --------
    {
        LapColumn<U2PITCH> col(&P.S.u[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < RJ; rr++) {
            q4 u, un, dn;
            a0[rr] = col.row(rr, u);
            if (rr == 0) cp_async_wait<0>();
            const q4 dv = ld4(&P.S.du[lz + rr + HALO][lx + HALO]), kv = ld4(&P.k[rr][tid].x);
            if constexpr (FULL) {
                dn = fma4(kv, a0[rr], dv);
                un = add4(u, dn);
            } else {
                if (rr == src >> 2) add_source(a0[rr], src & 3, A.c.wav[T.wav_off + n]);
                const q4 w = row_w(We, lx, lz, rr);
                dn = mul4(w, fma4(kv, a0[rr], dv));
                un = fma4(w, u, dn);
            }
            st4(&P.Vu[lz + rr + HALO][lx + HALO], un);
            if (core) st4(&P.du[rr][tid].x, dn);
        }
    }
    {
        LapColumn<U2PITCH> col(&P.S.p[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < RJ; rr++) {
            q4 p, pn, dn;
            const q4 ap = col.row(rr, p);
            const q4 dv = ld4(&P.S.dp[lz + rr + HALO][lx + HALO]), kv = ld4(&P.k[rr][tid].x);
            const q4 t = fma4(ld4(&P.dk[rr][tid].x), a0[rr], fma4(kv, ap, dv));
            if constexpr (FULL) {
                dn = t;
                pn = add4(p, dn);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                dn = mul4(w, t);
                pn = fma4(w, p, dn);
            }
            st4(&P.Vp[lz + rr + HALO][lx + HALO], pn);
            if (core) st4(&P.dp[rr][tid].x, dn);
        }
    }
    __syncthreads();  // u0^{n+1} and p^{n+1} complete; the stage is no longer read
    mid();

    // Receivers: sample n is p^{n+1} (the ring warps, free from here on).
    if (!core) {
        for (int e = T.rec_begin + tid - NCOREJ; e < T.rec_end; e += NTJ - NCOREJ) {
            const TileRec tr = A.c.recs[e];
            A.d[T.doff + (long long)n * T.nrec + tr.r] = P.Vp[tr.cell / TX + HALO][tr.cell % TX + HALO];
        }
    }
    if (!two) return;  // the record ends at n+1: the state is not needed any more

    // ---- step n+1 on the core ----------------------------------------------
    if (ok) {
        const long long cbase = T.foff + (long long)i0 * pitch + j;
        {
            LapColumn<VP> col(&P.Vu[lz][lx + HALO]);
#pragma unroll
            for (int rr = 0; rr < RJ; rr++) {
                q4 u, un, d2;
                a0[rr] = col.row(rr, u);
                const q4 kv = ld4(&P.k[rr][tid].x), dv = ld4(&P.du[rr][tid].x);
                if constexpr (FULL) {
                    d2 = fma4(kv, a0[rr], dv);
                    un = add4(u, d2);
                } else {
                    if (rr == src >> 2) add_source(a0[rr], src & 3, A.c.wav[T.wav_off + n + 1]);
                    const q4 w = row_w(We, lx, lz, rr);
                    d2 = mul4(w, fma4(kv, a0[rr], dv));
                    un = fma4(w, u, d2);
                }
                if (rr < nrow) {
                    const long long c = cbase + (long long)rr * pitch;
                    st4(A.du_out + c, d2);
                    st4(A.un + c, un);
                }
            }
        }
        LapColumn<VP> col(&P.Vp[lz][lx + HALO]);
#pragma unroll
        for (int rr = 0; rr < RJ; rr++) {
            q4 p, pn, d2;
            const q4 ap = col.row(rr, p);
            const q4 kv = ld4(&P.k[rr][tid].x), dv = ld4(&P.dp[rr][tid].x);
            const q4 t = fma4(ld4(&P.dk[rr][tid].x), a0[rr], fma4(kv, ap, dv));
            if constexpr (FULL) {
                d2 = t;
                pn = add4(p, d2);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                d2 = mul4(w, t);
                pn = fma4(w, p, d2);
            }
            if (rr < nrow) {
                const long long c = cbase + (long long)rr * pitch;
                st4(A.dp_out + c, d2);
                st4(A.pn + c, pn);
            }
        }
    }
    // Receivers: sample n+1 is p^{n+2}, read back from the pool.
    if (T.rec_end > T.rec_begin) sample_from_pool<NTJ>(A.c, T, A.pn, A.d, n + 1);
}

__global__ void __launch_bounds__(NTJ, 1) born_joint_kernel(BornArgs A, const __grid_constant__ TileMaps M, int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    JointSmem &P = *reinterpret_cast<JointSmem *>(smem_raw);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_pairs<kJointStageBytes, LEADERJ>(
        A.c, ntiles, PairLoopSmem{&P.S, P.We, &P.tail}, tid,
        [&](const TileInfo &N, unsigned bar) {
            tma_load_3d(smem_u32(&P.S.u), &M.m[0], N.x0 - HALO2, N.z0 - HALO2, N.slot, bar);
            tma_load_3d(smem_u32(&P.S.p), &M.m[1], N.x0 - HALO2, N.z0 - HALO2, N.slot, bar);
            tma_load_3d(smem_u32(&P.S.du), &M.m[2], N.x0 - HALO, N.z0 - HALO, N.slot, bar);
            tma_load_3d(smem_u32(&P.S.dp), &M.m[3], N.x0 - HALO, N.z0 - HALO, N.slot, bar);
        },
        [&](const TileInfo &N) {
            copy_item<RJ>(P.k, A.c.kap, A.c, N, tid);
            copy_item<RJ>(P.dk, A.dkap, A.c, N, tid);
        },
        [](int) {}, []() {},
        [&](const TileInfo &T, const TileEdge &We, auto mid) {
            const bool two = T.nt > A.n + 1;
            if (T.flags & TI_FULL2) joint_tile<true>(A, P, We, T, tid, two, mid);
            else joint_tile<false>(A, P, We, T, tid, two, mid);
        },
        [](int) {});
}

// ---------------------------------------------------------------------------
// Two-step adjoint: steps k (nu^{k+1} -> nu^k) and k-1 in one launch, the
// same layout and stage refill as fwd_pair_kernel.  The data of step k are
// added to the staged D_nu (inject_here) or already in it (D' = D + kappa
// r^{k-1}, launch_adj_inject); the data of step k-1 are added to the core's
// D_nu^k after step k.  The image accumulator
// takes a^{k-1} nu^k (tiles whose record reaches step k) and then a^{k-2}
// nu^{k-1}, in that order, as two one-step launches would.
// ---------------------------------------------------------------------------
template <bool FULL, class MidFn>
__device__ __forceinline__ void adj_pair_tile(const AdjArgs &A, Pair2Stage &S, VTile &V, ItemSlots &I, const TileEdge &We,
                                              const TileInfo &T, int tid, MidFn mid) {
    int lx, lz;
    item_of<R4>(tid, lx, lz);
    const bool core = tid < NCORE;
    const int k = A.k, pitch = T.pitch;
    const int j = T.x0 + lx, i0 = T.z0 + lz;
    const int nrow = FULL ? R4 : A.c.NZ - i0;
    const bool ok = core && (FULL || j < T.nxw);
    const long long cbase = T.foff + (long long)i0 * pitch + j;

    // ---- step k on the item --------------------------------------------------
    {
        LapColumn<U2PITCH> col(&S.u[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            q4 nu;
            const q4 a = col.row(rr, nu);
            if (rr == 0) cp_async_wait<0>();
            const q4 dv = ld4(&S.d[lz + rr + HALO][lx + HALO]);
            const q4 kv = ld4(&I.k[rr][tid].x);
            q4 nn, dn;
            if constexpr (FULL) {
                dn = fma4(kv, a, dv);
                nn = add4(nu, dn);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                dn = mul4(w, fma4(kv, a, dv));
                nn = fma4(w, nu, dn);
            }
            st4(&V[lz + rr + HALO][lx + HALO], nn);
            if (core) st4(&I.d[rr][tid].x, dn);
        }
    }
    // The image and the background terms of the second step (prefetched into
    // L2 a tile ahead), a row ahead of the arithmetic, the first requested
    // before the barrier.  a^{k-1} exists only where the record reaches step
    // k (a stored history holds the shots active at each step only).
    const bool image_k = T.nt > k - 1;
    q4 gq{}, a1q{}, a2q{};
    auto fetch = [&](int rr) {
        if (ok && rr < nrow) {
            const long long c = cbase + (long long)rr * pitch;
            gq = ld4(A.g + c);
            if (image_k) a1q = ld4(A.a + c);
            a2q = ld4(A.a2 + c);
        }
    };
    fetch(0);
    __syncthreads();  // nu^k and D_nu^k complete; the stage is no longer read
    // Data of step k-1 at the tile's receivers: D' = D_nu^k + kappa r^{k-2}.
    if (T.rec_end > T.rec_begin) {
        const float *rk = A.r + T.doff + (long long)(k - 2) * T.nrec;
        for (int e = T.rec_begin + tid; e < T.rec_end; e += NT2)
            if (e == T.rec_begin || A.c.recs[e - 1].cell != A.c.recs[e].cell) {
                const int z = A.c.recs[e].cell / TX, x = A.c.recs[e].cell % TX;
                const int item = (z / R4) * 16 + x / 4;
                const float kc = (&I.k[z % R4][item].x)[x % 4];
                float &d = (&I.d[z % R4][item].x)[x % 4];
                d = fmaf(kc, receiver_sum(A.c.recs, e, T.rec_end, rk), d);
            }
        __syncthreads();
    }
    mid();

    // ---- step k-1 on the core, imaging of both steps --------------------------
    if (!ok) return;
    LapColumn<VP> col(&V[lz][lx + HALO]);
#pragma unroll
    for (int rr = 0; rr < R4; rr++) {
        q4 nu;  // nu^k
        const q4 a = col.row(rr, nu);
        q4 g = gq;
        const q4 a1 = a1q, a2 = a2q;
        if (rr + 1 < R4) fetch(rr + 1);
        const q4 kv = ld4(&I.k[rr][tid].x), dn = ld4(&I.d[rr][tid].x);
        q4 d2, nn;
        if constexpr (FULL) {
            d2 = fma4(kv, a, dn);
            nn = add4(nu, d2);
        } else {
            const q4 w = row_w(We, lx, lz, rr);
            d2 = mul4(w, fma4(kv, a, dn));
            nn = fma4(w, nu, d2);
        }
        if (image_k) g = fma4(a1, nu, g);
        g = fma4(a2, nn, g);
        if (rr < nrow) {
            const long long c = cbase + (long long)rr * pitch;
            st4(A.dd_out + c, d2);
            st4(A.nun + c, nn);
            st4(A.g + c, g);
        }
    }
}

__global__ void __launch_bounds__(NT2, 2) adj_pair_kernel(AdjArgs A, const __grid_constant__ TileMaps M, int ntiles) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PairSmem<ItemSlots> P(smem_raw);
    InjBuf &IB = *reinterpret_cast<InjBuf *>(smem_raw + kPair2Smem);
    const int tid = threadIdx.x + threadIdx.y * 32;
    // Data of step k injected here (inject_here): warp 8, free in the second
    // step, lists the next tile's grown-region injection (kappa and the
    // receivers' summed data, from global memory) while the core warps run
    // that step; after the tile's stage lands every thread adds the list to
    // the staged D_nu, D' = fmaf(kappa, sum, D) as the separate pass computes
    // it.  Shots whose record ends before step k take none.
    const bool inj = A.inject_here && A.c.xrec_off != nullptr;
    const bool lister = inj && tid >= NCORE && tid < NCORE + 32;
    auto build = [&](int t) {
        if (!lister) return;
        const int lane = tid - NCORE;
        const int xb = A.c.xrec_off[t], xe = A.c.xrec_off[t + 1];
        const TileInfo &Tg = A.c.infos[t];
        const bool has = Tg.nt > A.k - 1;
        const float *rk = A.r + Tg.doff + (long long)(A.k - 1) * Tg.nrec;
        for (int e = xb + lane; has && e < xe; e += 32) {
            InjEntry en{-1, 0.f, 0.f};
            if (e == xb || A.c.xrecs[e - 1].cell != A.c.xrecs[e].cell) {
                const int cell = A.c.xrecs[e].cell, ez = cell / E, ex = cell % E;
                en.off = cell;
                en.kap = A.c.kap[(long long)Tg.mc * A.c.mstride + (long long)(Tg.z0 - HALO + ez) * A.c.pf + Tg.mx +
                                 ex - HALO];
                en.sum = receiver_sum(A.c.xrecs, e, xe, rk);
            }
            IB.e[e - xb] = en;
        }
        if (lane == 0) IB.n = has ? xe - xb : 0;
    };
    run_pairs<kPair2StageBytes, LEADER2>(
        A.c, ntiles, P.loop(), tid,
        // The same tile's image, a^{k-1} and a^{k-2}, which the second step
        // loads from global memory, are prefetched into L2 with the stage.
        [&](const TileInfo &N, unsigned bar) {
            tma_load_3d(smem_u32(&P.S.u), &M.m[0], N.x0 - HALO2, N.z0 - HALO2, N.slot, bar);
            tma_load_3d(smem_u32(&P.S.d), &M.m[1], N.x0 - HALO, N.z0 - HALO, N.slot, bar);
            tma_prefetch_l2_3d(&M.m[3], N.x0, N.z0, N.slot);
            tma_prefetch_l2_3d(&M.m[4], N.x0, N.z0, N.slot);
            tma_prefetch_l2_3d(&M.m[5], N.x0, N.z0, N.slot);
        },
        [&](const TileInfo &N) { copy_item<R4>(P.I.k, A.c.kap, A.c, N, tid); },
        build,
        [&]() {
            if (!inj) return;
            const int n = IB.n;  // uniform: written before the last barrier
            float *dflat = &P.S.d[0][0];
            for (int e = tid; e < n; e += NT2) {
                const InjEntry en = IB.e[e];
                if (en.off >= 0) dflat[en.off] = fmaf(en.kap, en.sum, dflat[en.off]);
            }
            if (n > 0) __syncthreads();
        },
        [&](const TileInfo &T, const TileEdge &We, auto mid) {
            if (T.flags & TI_INTERIOR2) adj_pair_tile<true>(A, P.S, P.V, P.I, We, T, tid, mid);
            else adj_pair_tile<false>(A, P.S, P.V, P.I, We, T, tid, mid);
        },
        build);
}

// D' = D_nu + kappa r^{k-1} at the receiver cells of the listed tiles (one
// CTA per tile; receivers sharing a cell summed in order, as in
// build_injection).
__global__ void adj_inject_kernel(AdjArgs A, const int *__restrict__ rtiles) {
    // Launched as a programmatic dependent: it may start before the step
    // kernel that writes D_nu has finished, so it waits for it here, and lets
    // the next step kernel start its prologue at once.
    griddep_wait();
    griddep_launch_dependents();
    const TileInfo &T = A.c.infos[rtiles[blockIdx.x]];
    const float *rk = A.r + T.doff + (long long)(A.k - 1) * T.nrec;
    for (int e = T.rec_begin + threadIdx.x; e < T.rec_end; e += blockDim.x)
        if (e == T.rec_begin || A.c.recs[e - 1].cell != A.c.recs[e].cell) {
            const int cell = A.c.recs[e].cell;
            const int z = T.z0 + cell / TX, lx = cell % TX;
            const float kap = A.c.kap[(long long)T.mc * A.c.mstride + (long long)z * A.c.pf + T.mx + lx];
            float *d = A.dd + T.foff + (long long)z * T.pitch + T.x0 + lx;
            *d = fmaf(kap, receiver_sum(A.c.recs, e, T.rec_end, rk), *d);
        }
}

template <typename K, typename Args>
void launch_pdl2(K kernel, int grid, const Args &a, const TileMaps &maps, int ntiles, cudaStream_t s,
                 size_t smem = kPair2Smem, int threads = NT2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(32, threads / 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, a, maps, ntiles);
}

int occupancy_of(const void *fn, size_t smem = kPair2Smem, int threads = NT2) {
    int n = 0;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem);
    return n < 1 ? 1 : n;
}

}  // namespace

void launch_adj_pair(const AdjArgs &a, int ntiles, const TileMaps &maps, cudaStream_t s) {
    if (ntiles <= 0) return;
    static int sms = 0, occ = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        occ = occupancy_of((const void *)adj_pair_kernel, kAdj2Smem);
    }
    const int cap = occ * sms;
    launch_pdl2(adj_pair_kernel, ntiles < cap ? ntiles : cap, a, maps, ntiles, s, kAdj2Smem);
}

void launch_adj_inject(const AdjArgs &a, const int *rtiles, int nrtiles, cudaStream_t s) {
    if (nrtiles <= 0) return;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nrtiles);
    cfg.blockDim = dim3(128);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, adj_inject_kernel, a, rtiles);
}

void launch_born_pair(const BornArgs &a, int ntiles, const TileMaps &maps, cudaStream_t s) {
    if (ntiles <= 0) return;
    static int sms = 0, occ = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        occ = occupancy_of((const void *)born_pair_kernel, kBorn2Smem);
    }
    const int cap = occ * sms;
    launch_pdl2(born_pair_kernel, ntiles < cap ? ntiles : cap, a, maps, ntiles, s, kBorn2Smem);
}

void launch_born_joint(const BornArgs &a, int ntiles, const TileMaps &maps, cudaStream_t s) {
    if (ntiles <= 0) return;
    static int sms = 0, occ = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        occ = occupancy_of((const void *)born_joint_kernel, sizeof(JointSmem), NTJ);
    }
    const int cap = occ * sms;
    launch_pdl2(born_joint_kernel, ntiles < cap ? ntiles : cap, a, maps, ntiles, s, sizeof(JointSmem), NTJ);
}

int fwd_pair_occupancy() {
    const int a = occupancy_of((const void *)fwd_pair_kernel<ST_A>);
    const int b = occupancy_of((const void *)fwd_pair_kernel<ST_NONE>);
    const int c = occupancy_of((const void *)fwd_pair_kernel<ST_CK>);
    return a < b ? (a < c ? a : c) : (b < c ? b : c);
}

void launch_fwd_pair(const FwdArgs &a, int ntiles, const TileMaps &maps, cudaStream_t s) {
    if (ntiles <= 0) return;
    static int sms = 0, occ = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        occ = fwd_pair_occupancy();
    }
    const int cap = occ * sms;
    const int grid = ntiles < cap ? ntiles : cap;
    if (a.a_out) launch_pdl2(fwd_pair_kernel<ST_A>, grid, a, maps, ntiles, s);
    else if (a.ck_u) launch_pdl2(fwd_pair_kernel<ST_CK>, grid, a, maps, ntiles, s);
    else launch_pdl2(fwd_pair_kernel<ST_NONE>, grid, a, maps, ntiles, s);
}

}  // namespace dhfwi
