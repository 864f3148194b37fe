// Two-step (time-blocked) forward, adjoint and Born kernels for sm_103a: a tile
// advances by two steps of the recurrence of Section 2.1 (Eq. 1, summed form;
// see fd_kernels.cu) at a time, so u and D cross HBM once per two updates.
//
// One cooperative launch takes many step pairs (run_flow): its CTAs walk the
// items (pair m, tile) in that order, and an item waits only for the pair m-1
// of the tile and its up to eight neighbours, not for the whole grid.  A launch
// per pair left 15 % of the SM time idle at 32 shots of 400 x 1200 (an unfilled
// last wave, launch, prologue).  Plans whose tiles are all resident at once still
// take a launch per pair (api.cu, flow_pairs).
//
// Per 64 x 64 tile the TMA stages u^n with an 8-cell halo and D^n with a
// 4-cell ring.  Step n is computed on the tile and its ring, giving
// u^{n+1} in shared memory (zero outside the window: the Dirichlet boundary);
// step n+1 is then computed on the core from it.  The ring cells are
// recomputed by each tile that needs them (1024 per 4096, the corners, which
// no stencil reaches, left out), so tiles exchange data only between pairs;
// since they read D^n on their neighbours' cells, u and D alternate between two
// pools each.  Every cell goes through the same floating-point operations in
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
// What bounds it: latency at 20 warps per SM (FMA pipe half busy).  64 shots of
// 400 x 1200, ms per pass of 3983 steps:
//   forward 128.7 (two columns x 9 rows per thread, sponge factors and bounds
//     tests computed per row) -> 117.7 (items, kappa and sponge factors loaded
//     where they are used) -> 97.0 (both copied a tile ahead) -> 94.9 (kappa
//     awaited only where it is used, after the first Laplacian) -> 91.5 (many
//     pairs per launch); storing a^n 135 -> 116 -> 109 -> 108;
//   adjoint 163 -> 153 -> 148 -> 135;
//   16 shots (2.7 tiles per resident CTA), forward with the store and adjoint:
//     91.5 -> 77.7 -> 76.0 -> 63.4.
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

#include <algorithm>

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
// An item of a launch: a tile and its step pair.
struct FlowItem {
    TileInfo T;
    int m, tile;  // pair of the launch (-1: no more items), tile of the plan
    int n;        // first step of the pair (forward, Born: n, then n+1; adjoint: k, then k-1)
    int need;     // pairs that the tile and its neighbours must have done
    float *p[6];  // per kernel: arrays at the tile's first cell
    float *row;   // the shot's record row of step n (adjoint: r^{k-1})
    int two;      // whether the shot records past step n
    int eager;    // published as soon as it is done (see run_flow)
    int ready;    // its dependencies have been seen to be done
    int pad[3];
};
static_assert(sizeof(FlowItem) % 16 == 0, "16-byte copies of the tile's descriptor");
// The stage's barrier, the items of this tile, the next one (whose loads the
// leader warp issues in the middle of this one) and the one after, and the
// leader warp's place in the sequence.
struct PairTail {
    unsigned long long bar[2];
    FlowItem item[3];
    int wm, wi, pad[2];
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
        cp_async16(&slots[rr][tid], m + model_row(T.z0 + lz + rr, c.NZ, c.pf));
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

// ---------------------------------------------------------------------------
// The item loop.  CTA b takes the items b, b + gridDim.x, ... of the sequence
// of pairs m = 0, 1, ... with count(m) tiles each (shots by record length, so
// the active ones are a prefix).  The launch is
// cooperative, so all CTAs are resident; items are taken in order, so the
// first unfinished one never waits for a later one, and every wait ends.
//
// done[tile] counts the pairs of a tile that are complete in memory.  An item's
// tensor loads wait until the tile and its neighbours have done the pair
// before (they also have read what the item overwrites by then).  An item of a
// pair with few tiles is published (fence, release) as soon as its stores are
// issued; one of a pair with two or more tiles per CTA in the middle of the CTA's
// next item, when the stores have long drained and the fence delays no one, and
// nobody waits for the flag yet (from two tiles per CTA on: 16 and 20 shots of
// 400 x 1200, gradient, 64.4 -> 60.6 and 77.7 -> 72.0 ms against from four on).
// That deferral cannot deadlock: what depends on such an item comes more than
// gridDim.x items after it, the CTA's next item gridDim.x after it, so the next
// item depends (through any chain) only on deferred items before this one, which
// are published first.
//
// One stage, refilled in the middle of a tile so that the next tile's loads
// overlap step n+1; the barrier that opens a tile also certifies that every
// thread is done with the tile before.  Waits are bounded as in run_tiles: a
// CTA whose loads or dependencies do not come within about a second sets
// *tflag and leaves, and the others that wait for it leave too.
//
// BYTES: the stage's; NC: core threads; LEADER: first thread of the leader
// warp, a ring warp like the one before it (the publishing one).  K gives
//   count(m), step(m), need(m, T): the sequence (see FlowItem);
//   ptr(i, m, T), row(m, T): an item's arrays;
//   issue(item, bar): the leader's tensor loads of an item's stage; prefetch
//     (item, lane): the leader warp's L2 prefetches for it;
//   fill(item): every thread's copies of a tile's model values into its slots
//     (body awaits them with cp_async_wait<0>() before their first use: no
//     other thread reads them, so their latency overlaps the opening barrier
//     and the first Laplacian);
//   begin(item): before the first tile, no barrier inside;
//   open(item): once a tile's stage has landed (may synchronise the CTA);
//   body(item, We, mid): the tile, calling mid() after the barrier that ends
//     step n (the stage is no longer read then: the leader refills it);
//   close(item): after the tile, with the next one.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned *p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Orders generic-proxy accesses to global memory with async-proxy ones (TMA).
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
// Named barriers: id 1 the core and the publishing warp, id 2 the core.
template <int ID, int N>
__device__ __forceinline__ void bar_sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }
template <int ID, int N>
__device__ __forceinline__ void bar_arrive() { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(N) : "memory"); }

// Leader warp: whether the item's tile and its neighbours have done `need`
// pairs; with wait, waits for it (bounded) and returns false when it did not
// come.  True orders the loads that follow, of any lane, after their stores.
__device__ __forceinline__ bool deps_done(const FlowArgs &F, const StepCommon &c, const FlowItem &it, int lane,
                                          bool wait) {
    if (it.need == 0) return true;
    const int ntx = (it.T.nxw + TX - 1) / TX, ntz = (c.NZ + TZ - 1) / TZ;
    const int dz = lane / 3 - 1, dx = lane % 3 - 1;
    const int tz = it.T.z0 / TZ + dz, tx = it.T.x0 / TX + dx;
    const bool mine = lane < 9 && tz >= 0 && tz < ntz && tx >= 0 && tx < ntx;
    const unsigned *p = F.done + it.tile + dz * ntx + dx;
    const unsigned need = (unsigned)it.need;
    bool ok = __all_sync(0xffffffffu, !mine || ld_acquire(p) >= need);
    if (!ok && wait) {
        const unsigned long long t0 = global_ns();
        for (int spin = 1; !(ok = __all_sync(0xffffffffu, !mine || ld_acquire(p) >= need)); spin++)
            if ((spin & 63) == 0) {
                const bool stop = lane == 0 && (global_ns() - t0 > 1000000000ull || ld_acquire(c.tflag) != 0u);
                if (__any_sync(0xffffffffu, stop)) return false;
            }
    }
    __syncwarp();  // the vote orders no memory: every lane's acquire before what any lane does next
    return ok;
}

template <unsigned BYTES, int NC, int LEADER, class K>
__device__ __forceinline__ void run_flow(const FlowArgs &F, const StepCommon &c, const PairLoopSmem &P, int tid,
                                         const K &k) {
    const bool lead = tid >= LEADER, leader = tid == LEADER, pub = tid >= LEADER - 32 && !lead;
    const int lane = tid & 31;
    int pub_tile = -1;  // publishing warp: the item before, if not published yet
    unsigned pub_val = 0;
    const unsigned bar = smem_u32(&P.tail->bar[0]);
    if (smem_u32(P.stage) & 127u) {
        if (leader) atomicExch(c.tflag, 2u);
        return;
    }
    // Leader warp: the next item of the CTA's sequence into `it`.
    auto take = [&](FlowItem &it, bool advance) {
        int m = P.tail->wm, i = P.tail->wi;
        if (advance) i += gridDim.x;
        int cnt = 0;
        while (m < F.npairs && i >= (cnt = k.count(m))) {
            i -= cnt;
            m++;
        }
        __syncwarp();
        if (lane == 0) {
            P.tail->wm = m;
            P.tail->wi = i;
        }
        if (m >= F.npairs) {
            if (lane == 0) it.m = -1;
            __syncwarp();
            return;
        }
        if (lane < 5)
            reinterpret_cast<int4 *>(&it.T)[lane] = __ldg(reinterpret_cast<const int4 *>(&c.infos[i]) + lane);
        __syncwarp();
        const TileInfo &T = it.T;
        if (lane < 6) it.p[lane] = k.ptr(lane, m, T);
        if (lane == 6) {
            const int n = k.step(m);
            it.m = m;
            it.tile = i;
            it.n = n;
            it.need = k.need(m, T);
            it.row = k.row(m, T);
            it.two = T.nt > n + 1;
            it.eager = cnt < 2 * (int)gridDim.x + T.pitch / TX + 2;  // (neighbours: up to a tile row + 1 apart)
        }
        __syncwarp();
    };
    // Leader warp: an item's loads.
    auto load = [&](const FlowItem &it) {
        if (lane == 0) {
            // Between other CTAs' stores (seen by deps_done) and the tensor
            // loads of them, another proxy's.
            fence_proxy_async_global();
            fence_proxy_async();
            mbar_expect_tx(bar, BYTES);
            k.issue(it, bar);
        }
        k.prefetch(it, lane);
    };
    // One thread, after a barrier with the core: the item's stores before the flag.
    auto publish = [&](int tile, unsigned pairs) {
        if (F.npairs > 1) st_release(F.done + tile, pairs);
    };
    if (lead) {
        if (lane == 0) {
            mbar_init(bar, 1);
            fence_mbar_init();
            P.tail->wm = 0;
            P.tail->wi = blockIdx.x;
        }
        __syncwarp();
        take(P.tail->item[0], false);
        if (lane == 0) P.tail->item[0].ready = P.tail->item[1].ready = 0;
        __syncwarp();
        if (P.tail->item[0].m >= 0) take(P.tail->item[1], true);
    }
    __syncthreads();
    if (P.tail->item[0].m < 0) return;
    if (lead) copy_edge(P.We[0], c, P.tail->item[0].T, lane);
    cp_async_commit();
    k.fill(P.tail->item[0]);
    cp_async_commit();
    // Launches of one pair follow one another as programmatic dependents: up to
    // here only data older than the launch before was read.
    griddep_wait();
    griddep_launch_dependents();
    if (lead) {
        if (deps_done(F, c, P.tail->item[0], lane, true)) load(P.tail->item[0]);
        else if (lane == 0) atomicExch(c.tflag, 1u);
    }
    k.begin(P.tail->item[0]);
    unsigned phase = 0;
    int slot = 0, next = 1;
    for (;;) {
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
        const FlowItem &it = P.tail->item[slot];
        k.open(it);
        const bool more = P.tail->item[next].m >= 0;
        const int after = 3 - slot - next;
        // After a barrier: every thread is done with the stage.  The leader
        // warp refills it and looks ahead, the publishing warp publishes a
        // deferred item; both have to be back before the core is done.
        auto mid = [&]() {
            if (pub && lane == 0 && pub_tile >= 0) publish(pub_tile, pub_val);
            if (!lead || !more) return;
            const FlowItem &coming = P.tail->item[next];
            FlowItem &other = P.tail->item[after];
            const bool ready = coming.ready || deps_done(F, c, coming, lane, false);
            if (ready) load(coming);
            copy_edge(P.We[phase], c, coming.T, lane);
            take(other, true);
            if (!ready) {
                if (deps_done(F, c, coming, lane, true)) load(coming);
                else if (lane == 0) atomicExch(c.tflag, 1u);
            }
            // Whether the loads of the item after the next one can be issued
            // without a look at the flags then (a look costs the latency of L2,
            // which the refill of the stage would wait for).
            const bool r2 = other.m >= 0 && !other.eager && deps_done(F, c, other, lane, false);
            if (lane == 0) other.ready = r2;
            __syncwarp();
        };
        k.body(it, P.We[phase ^ 1u], mid);
        if (tid < NC) {
            if (it.eager) bar_arrive<1, NC + 32>();
        } else if (pub) {
            pub_tile = it.eager ? -1 : it.tile;
            pub_val = (unsigned)it.need + 1u;
            if (it.eager) {
                bar_sync<1, NC + 32>();
                if (lane == 0) publish(it.tile, pub_val);
            }
        }
        cp_async_commit();  // (the copies of mid())
        if (!more) break;
        k.fill(P.tail->item[next]);
        k.close(P.tail->item[next]);
        cp_async_commit();
        slot = next;
        next = after;
    }
    __syncthreads();
    if (pub && lane == 0 && pub_tile >= 0) publish(pub_tile, pub_val);  // the last item
}

// Receivers of a tile: sample n from u^{n+1} in shared memory, by the ring
// threads (free after the first step); sample n+1 from the core's stores, by
// the core threads.
template <int NC, int NT>
__device__ __forceinline__ void sample_first(const StepCommon &c, const FlowItem &it, const VTile &V, int tid) {
    for (int e = it.T.rec_begin + tid - NC; e < it.T.rec_end; e += NT - NC) {
        const TileRec tr = c.recs[e];
        it.row[tr.r] = V[tr.cell / TX + HALO][tr.cell % TX + HALO];
    }
}
template <int NC>
__device__ __forceinline__ void sample_second(const StepCommon &c, const FlowItem &it, const float *f, int tid) {
    if (it.T.rec_end <= it.T.rec_begin) return;
    bar_sync<2, NC>();
    for (int e = it.T.rec_begin + tid; e < it.T.rec_end; e += NC) {
        const TileRec tr = c.recs[e];
        it.row[it.T.nrec + tr.r] = f[(tr.cell / TX) * it.T.pitch + tr.cell % TX];
    }
}

// Forward: STORE says what else a launch stores (nothing, a^n and a^{n+1}, or
// the checkpoint u^n, D^n).  Item arrays: u^{n+2}, D^{n+2}, a^n, a^{n+1},
// checkpoint u and D (null: none at this step).
enum { ST_NONE = 0, ST_A = 1, ST_CK = 2 };
template <int STORE, bool FULL, class MidFn>
__device__ __forceinline__ void pair_tile(const FwdFlow &A, const Pair2Stage &S, VTile &V, ItemSlots &I,
                                          const TileEdge &We, const FlowItem &it, int tid, MidFn mid) {
    const TileInfo &T = it.T;
    int lx, lz;
    item_of<R4>(tid, lx, lz);
    const bool core = tid < NCORE;
    const int nrow = FULL ? R4 : A.c.NZ - (T.z0 + lz);
    const bool ok = core && (FULL || T.x0 + lx < T.nxw);
    const int src = FULL ? -1 : item_source<R4>(T, lx, lz);
    const int off = lz * T.pitch + lx;

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
                if (rr == src >> 2) add_source(a, src & 3, A.c.wav[T.wav_off + it.n]);
                const q4 w = row_w(We, lx, lz, rr);
                dn = mul4(w, fma4(kv, a, dv));
                un = fma4(w, u, dn);
            }
            st4(&V[lz + rr + HALO][lx + HALO], un);
            if (core) st4(&I.d[rr][tid].x, dn);
            if (STORE != ST_NONE && ok && rr < nrow) {
                const int o = off + rr * T.pitch;
                if constexpr (STORE == ST_CK) {
                    if (it.p[4]) {
                        st4(it.p[4] + o, u);
                        st4(it.p[5] + o, dv);
                    }
                }
                if constexpr (STORE == ST_A) st4(it.p[2] + o, a);
            }
        }
    }
    __syncthreads();  // u^{n+1} complete; the stage is no longer read
    mid();
    if (A.rec && !core) sample_first<NCORE, NT2>(A.c, it, V, tid);

    // ---- step n+1 on the core ----------------------------------------------
    if (!it.two || !core) return;  // (a record that ends at n+1 needs no further state)
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
                if (rr == src >> 2) add_source(a, src & 3, A.c.wav[T.wav_off + it.n + 1]);
                const q4 w = row_w(We, lx, lz, rr);
                d2 = mul4(w, fma4(kv, a, dn));
                un = fma4(w, u, d2);
            }
            if (rr < nrow) {
                const int o = off + rr * T.pitch;
                st4(it.p[1] + o, d2);
                st4(it.p[0] + o, un);
                if constexpr (STORE == ST_A) st4(it.p[3] + o, a);
            }
        }
    }
    if (A.rec) sample_second<NCORE>(A.c, it, it.p[0], tid);
}

// What the kernels of one field share: the sequence of a forward-time launch
// (pairs n0 + 2 m) and the arrays' addresses.
__device__ __forceinline__ long long cell0(const TileInfo &T) { return T.foff + (long long)T.z0 * T.pitch + T.x0; }
__device__ __forceinline__ int active_count(const FlowArgs &F, int n) {
    return min(__ldg(F.act + n), F.nt);
}
// a^n of a launch: a stored history's step, or a slot of a segment buffer.
__device__ __forceinline__ float *a_at(const ASteps &a, int n) {
    return a.base + (a.off ? __ldg(a.off + min(n, a.last)) : (long long)(n - a.first) * a.stride);
}
// L2 prefetch of a tile's rows (64 columns: two lines each), by one warp.
__device__ __forceinline__ void prefetch_rows(const float *f, const TileInfo &T, int NZ, int lane) {
    const float *p = f + (long long)(lane >> 1) * T.pitch + 32 * (lane & 1);
#pragma unroll
    for (int r = 0; r < TZ; r += 16)
        if (T.z0 + r + (lane >> 1) < NZ)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p + (long long)r * T.pitch) : "memory");
}

template <int STORE>
struct FwdK {
    const FwdFlow &A;
    const TileMaps &M;
    const PairSmem<ItemSlots> &P;
    int tid;
    __device__ __forceinline__ int step(int m) const { return A.n0 + 2 * m; }
    __device__ __forceinline__ int count(int m) const { return active_count(A.f, step(m)); }
    __device__ __forceinline__ int need(int m, const TileInfo &) const { return m; }
    __device__ __forceinline__ float *ptr(int i, int m, const TileInfo &T) const {
        const int n = step(m);
        const long long c = cell0(T);
        if (i < 2) return (i == 0 ? A.u[(m + 1) & 1] : A.d[(m + 1) & 1]) + c;
        if (STORE == ST_A && i < 4) return a_at(A.a, n + i - 2) + c;
        if (STORE == ST_CK && i >= 4 && n % A.ck_every == 0)
            return A.ck + (2 * (long long)(n / A.ck_every - A.ck_first) + i - 4) * A.pool + c;
        return nullptr;
    }
    __device__ __forceinline__ float *row(int m, const TileInfo &T) const {
        return A.rec + T.doff + (long long)step(m) * T.nrec;
    }
    __device__ __forceinline__ void issue(const FlowItem &it, unsigned bar) const {
        const TileInfo &T = it.T;
        tma_load_3d(smem_u32(&P.S.u), &M.m[it.m & 1], T.x0 - HALO2, T.z0 - HALO2, T.slot, bar);
        tma_load_3d(smem_u32(&P.S.d), &M.m[2 + (it.m & 1)], T.x0 - HALO, T.z0 - HALO, T.slot, bar);
    }
    __device__ __forceinline__ void prefetch(const FlowItem &, int) const {}
    __device__ __forceinline__ void fill(const FlowItem &it) const { copy_item<R4>(P.I.k, A.c.kap, A.c, it.T, tid); }
    __device__ __forceinline__ void begin(const FlowItem &) const {}
    __device__ __forceinline__ void open(const FlowItem &) const {}
    __device__ __forceinline__ void close(const FlowItem &) const {}
    template <class MidFn>
    __device__ __forceinline__ void body(const FlowItem &it, const TileEdge &We, MidFn mid) const {
        if (it.T.flags & TI_FULL2) pair_tile<STORE, true>(A, P.S, P.V, P.I, We, it, tid, mid);
        else pair_tile<STORE, false>(A, P.S, P.V, P.I, We, it, tid, mid);
    }
};

template <int STORE>
__global__ void __launch_bounds__(NT2, 2)
    fwd_pair_kernel(const __grid_constant__ FwdFlow A, const __grid_constant__ TileMaps M) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PairSmem<ItemSlots> P(smem_raw);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_flow<kPair2StageBytes, NCORE, LEADER2>(A.f, A.c, P.loop(), tid, FwdK<STORE>{A, M, P, tid});
}

// ---------------------------------------------------------------------------
// Two-step Born from a^n (see born_hist_tma_kernel): the scattered field p
// advances by the steps n and n+1 with the background terms a^n and a^{n+1} of
// a stored forward pass.  The layout
// of fwd_pair_kernel, with d kappa in slots beside kappa; a^n, read once per
// step, is prefetched into L2 a tile ahead and loaded a row ahead.
// ---------------------------------------------------------------------------
// Item arrays: p^{n+2}, D_p^{n+2}, a^n, a^{n+1}.
template <bool FULL, class MidFn>
__device__ __forceinline__ void born_pair_tile(const BornFlow &A, const PairSmem<BornSlots> &P, const TileEdge &We,
                                               const FlowItem &it, int tid, MidFn mid) {
    const TileInfo &T = it.T;
    int lx, lz;
    item_of<R4>(tid, lx, lz);
    const bool core = tid < NCORE;
    const int NZ = A.c.NZ, j = T.x0 + lx, i0 = T.z0 + lz;
    const int nrow = FULL ? R4 : NZ - i0;
    const bool ok = core && (FULL || j < T.nxw);
    const int off = lz * T.pitch + lx;
    // a outside the window reads as zero (its padding columns may hold anything).
    const bool in_x = FULL || (j >= 0 && j < T.nxw);
    auto load_a = [&](const float *a, int rr) {
        if (FULL) return ld4(a + off + rr * T.pitch);
        q4 v{0ull, 0ull};
        if (in_x && (unsigned)(i0 + rr) < (unsigned)NZ) {
            v = ld4(a + off + rr * T.pitch);
            const int w = T.nxw - j;  // columns of the quad inside the window
            if (w < 4) v = q4{w < 2 ? keep_lo(v.lo, false) : v.lo, w < 3 ? 0ull : keep_lo(v.hi, false)};
        }
        return v;
    };

    q4 dn[R4];

    // ---- step n on the item ------------------------------------------------
    {
        q4 an = load_a(it.p[2], 0);
        LapColumn<U2PITCH> col(&P.S.u[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            const q4 a0 = an;
            if (rr + 1 < R4) an = load_a(it.p[2], rr + 1);
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

    if (!core) sample_first<NCORE, NT2>(A.c, it, P.V, tid);
    if (!it.two || !core) return;  // (a record that ends at n+1 needs no further state)

    // ---- step n+1 on the core ----------------------------------------------
    if (ok) {
        q4 an = load_a(it.p[3], 0);
        LapColumn<VP> col(&P.V[lz][lx + HALO]);
#pragma unroll
        for (int rr = 0; rr < R4; rr++) {
            const q4 a0 = an;
            if (rr + 1 < R4) an = load_a(it.p[3], rr + 1);
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
                const int o = off + rr * T.pitch;
                st4(it.p[1] + o, d2);
                st4(it.p[0] + o, pn);
            }
        }
    }
    sample_second<NCORE>(A.c, it, it.p[0], tid);
}

struct BornK {
    const BornFlow &A;
    const TileMaps &M;
    const PairSmem<BornSlots> &P;
    int tid;
    __device__ __forceinline__ int step(int m) const { return A.n0 + 2 * m; }
    __device__ __forceinline__ int count(int m) const { return active_count(A.f, step(m)); }
    __device__ __forceinline__ int need(int m, const TileInfo &) const { return m; }
    __device__ __forceinline__ float *ptr(int i, int m, const TileInfo &T) const {
        const long long c = cell0(T);
        if (i < 2) return (i == 0 ? A.p[(m + 1) & 1] : A.dp[(m + 1) & 1]) + c;
        return i < 4 ? a_at(A.a, step(m) + i - 2) + c : nullptr;
    }
    __device__ __forceinline__ float *row(int m, const TileInfo &T) const {
        return A.rec + T.doff + (long long)step(m) * T.nrec;
    }
    __device__ __forceinline__ void issue(const FlowItem &it, unsigned bar) const {
        const TileInfo &T = it.T;
        tma_load_3d(smem_u32(&P.S.u), &M.m[it.m & 1], T.x0 - HALO2, T.z0 - HALO2, T.slot, bar);
        tma_load_3d(smem_u32(&P.S.d), &M.m[2 + (it.m & 1)], T.x0 - HALO, T.z0 - HALO, T.slot, bar);
    }
    __device__ __forceinline__ void prefetch(const FlowItem &it, int lane) const {
        prefetch_rows(it.p[2], it.T, A.c.NZ, lane);
        if (it.two) prefetch_rows(it.p[3], it.T, A.c.NZ, lane);
    }
    __device__ __forceinline__ void fill(const FlowItem &it) const {
        copy_item<R4>(P.I.k, A.c.kap, A.c, it.T, tid);
        copy_item<R4>(P.I.dk, A.dkap, A.c, it.T, tid);
    }
    __device__ __forceinline__ void begin(const FlowItem &) const {}
    __device__ __forceinline__ void open(const FlowItem &) const {}
    __device__ __forceinline__ void close(const FlowItem &) const {}
    template <class MidFn>
    __device__ __forceinline__ void body(const FlowItem &it, const TileEdge &We, MidFn mid) const {
        if (it.T.flags & TI_INTERIOR2) born_pair_tile<true>(A, P, We, it, tid, mid);
        else born_pair_tile<false>(A, P, We, it, tid, mid);
    }
};

__global__ void __launch_bounds__(NT2, 2)
    born_pair_kernel(const __grid_constant__ BornFlow A, const __grid_constant__ TileMaps M) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PairSmem<BornSlots> P(smem_raw);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_flow<kPair2StageBytes, NCORE, LEADER2>(A.f, A.c, P.loop(), tid, BornK{A, M, P, tid});
}

// ---------------------------------------------------------------------------
// Two-step Born, both fields (see born_tma_kernel): u0 and p advance by the
// steps n and n+1 in one launch, so each field crosses HBM once per two steps
// (16 bytes per cell and step of both, where the one-step kernel moves 32) and
// a^n stays in registers between the two updates of a cell.  Both fields' stages
// fill most of the shared memory, so one CTA takes a tile, and a thread may hold
// twice the registers of the other two-step kernels: items of 4 x 4 cells (256 of
// the core, 64 of the ring), both D of the core in registers between the steps,
// only kappa and its perturbation in slots.  Bound by latency at 10 warps per SM.
// 64 shots of 400 x 1200, 3983 steps: 272 ms (one step per launch, DRAM 64 % busy)
// -> 222.5 with items of 4 x 2 cells (20 warps, D in slots) -> 218.4 with these; 30
// shots 105.6 -> 102.7, 8 shots 29.3 -> 27.4, 4 shots of 101 x 101 (36 tiles, latency
// of a step only) 1.90 -> 1.83; 4 x 4 with D in slots 102.0, 28.1 and 1.92.
// A forward pair launch that stores a^n and a scattered-field one that reads it
// (24 bytes) took 270 ms.
// ---------------------------------------------------------------------------
constexpr int RJ = 4, NTJ = 320, NCOREJ = 256, LEADERJ = 288;
struct JointStage {
    float u[U2R][U2PITCH], p[U2R][U2PITCH];
    float du[E][E], dp[E][E];
};
constexpr unsigned kJointStageBytes = sizeof(JointStage);
struct JointSmem {
    JointStage S;
    VTile Vu, Vp;
    float4 k[RJ][NTJ], dk[RJ][NTJ];  // per-thread slots, see ItemSlots
    TileEdge We[2];
    PairTail tail;
};
static_assert(sizeof(JointStage) == 8 * (U2R * U2PITCH + E * E) && sizeof(JointSmem) % 16 == 0, "stage layout");

// Item arrays: u0^{n+2}, D_u0^{n+2}, p^{n+2}, D_p^{n+2}.
template <bool FULL, class MidFn>
__device__ __forceinline__ void joint_tile(const BornFlow &A, JointSmem &P, const TileEdge &We, const FlowItem &it,
                                           int tid, MidFn mid) {
    const TileInfo &T = it.T;
    int lx, lz;
    item_of<RJ>(tid, lx, lz);
    const bool core = tid < NCOREJ;
    const int nrow = FULL ? RJ : A.c.NZ - (T.z0 + lz);
    const bool ok = core && (FULL || T.x0 + lx < T.nxw);
    const int off = lz * T.pitch + lx;
    const int src = FULL ? -1 : item_source<RJ>(T, lx, lz);
    q4 a0[RJ], du[RJ], dp[RJ];

    // ---- step n on the item: the background, then the scattered field --------
    {
        LapColumn<U2PITCH> col(&P.S.u[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < RJ; rr++) {
            q4 u, un;
            a0[rr] = col.row(rr, u);
            if (rr == 0) cp_async_wait<0>();
            const q4 dv = ld4(&P.S.du[lz + rr + HALO][lx + HALO]), kv = ld4(&P.k[rr][tid].x);
            if constexpr (FULL) {
                du[rr] = fma4(kv, a0[rr], dv);
                un = add4(u, du[rr]);
            } else {
                if (rr == src >> 2) add_source(a0[rr], src & 3, A.c.wav[T.wav_off + it.n]);
                const q4 w = row_w(We, lx, lz, rr);
                du[rr] = mul4(w, fma4(kv, a0[rr], dv));
                un = fma4(w, u, du[rr]);
            }
            st4(&P.Vu[lz + rr + HALO][lx + HALO], un);
        }
    }
    {
        LapColumn<U2PITCH> col(&P.S.p[lz + HALO][lx + HALO2]);
#pragma unroll
        for (int rr = 0; rr < RJ; rr++) {
            q4 p, pn;
            const q4 ap = col.row(rr, p);
            const q4 dv = ld4(&P.S.dp[lz + rr + HALO][lx + HALO]), kv = ld4(&P.k[rr][tid].x);
            const q4 t = fma4(ld4(&P.dk[rr][tid].x), a0[rr], fma4(kv, ap, dv));
            if constexpr (FULL) {
                dp[rr] = t;
                pn = add4(p, dp[rr]);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                dp[rr] = mul4(w, t);
                pn = fma4(w, p, dp[rr]);
            }
            st4(&P.Vp[lz + rr + HALO][lx + HALO], pn);
        }
    }
    __syncthreads();  // u0^{n+1} and p^{n+1} complete; the stage is no longer read
    mid();

    if (!core) sample_first<NCOREJ, NTJ>(A.c, it, P.Vp, tid);
    if (!it.two || !core) return;  // (a record that ends at n+1 needs no further state)

    // ---- step n+1 on the core ----------------------------------------------
    if (ok) {
        {
            LapColumn<VP> col(&P.Vu[lz][lx + HALO]);
#pragma unroll
            for (int rr = 0; rr < RJ; rr++) {
                q4 u, un, d2;
                a0[rr] = col.row(rr, u);
                const q4 kv = ld4(&P.k[rr][tid].x);
                if constexpr (FULL) {
                    d2 = fma4(kv, a0[rr], du[rr]);
                    un = add4(u, d2);
                } else {
                    if (rr == src >> 2) add_source(a0[rr], src & 3, A.c.wav[T.wav_off + it.n + 1]);
                    const q4 w = row_w(We, lx, lz, rr);
                    d2 = mul4(w, fma4(kv, a0[rr], du[rr]));
                    un = fma4(w, u, d2);
                }
                if (rr < nrow) {
                    const int o = off + rr * T.pitch;
                    st4(it.p[1] + o, d2);
                    st4(it.p[0] + o, un);
                }
            }
        }
        LapColumn<VP> col(&P.Vp[lz][lx + HALO]);
#pragma unroll
        for (int rr = 0; rr < RJ; rr++) {
            q4 p, pn, d2;
            const q4 ap = col.row(rr, p);
            const q4 kv = ld4(&P.k[rr][tid].x);
            const q4 t = fma4(ld4(&P.dk[rr][tid].x), a0[rr], fma4(kv, ap, dp[rr]));
            if constexpr (FULL) {
                d2 = t;
                pn = add4(p, d2);
            } else {
                const q4 w = row_w(We, lx, lz, rr);
                d2 = mul4(w, t);
                pn = fma4(w, p, d2);
            }
            if (rr < nrow) {
                const int o = off + rr * T.pitch;
                st4(it.p[3] + o, d2);
                st4(it.p[2] + o, pn);
            }
        }
    }
    sample_second<NCOREJ>(A.c, it, it.p[2], tid);
}

struct JointK {
    const BornFlow &A;
    const TileMaps &M;
    JointSmem &P;
    int tid;
    __device__ __forceinline__ int step(int m) const { return A.n0 + 2 * m; }
    __device__ __forceinline__ int count(int m) const { return active_count(A.f, step(m)); }
    __device__ __forceinline__ int need(int m, const TileInfo &) const { return m; }
    __device__ __forceinline__ float *ptr(int i, int m, const TileInfo &T) const {
        const int o = (m + 1) & 1;
        return i < 4 ? (i == 0 ? A.u[o] : i == 1 ? A.du[o] : i == 2 ? A.p[o] : A.dp[o]) + cell0(T) : nullptr;
    }
    __device__ __forceinline__ float *row(int m, const TileInfo &T) const {
        return A.rec + T.doff + (long long)step(m) * T.nrec;
    }
    __device__ __forceinline__ void issue(const FlowItem &it, unsigned bar) const {
        const TileInfo &T = it.T;
        const int i = it.m & 1;
        tma_load_3d(smem_u32(&P.S.u), &M.m[i], T.x0 - HALO2, T.z0 - HALO2, T.slot, bar);
        tma_load_3d(smem_u32(&P.S.p), &M.m[2 + i], T.x0 - HALO2, T.z0 - HALO2, T.slot, bar);
        tma_load_3d(smem_u32(&P.S.du), &M.m[4 + i], T.x0 - HALO, T.z0 - HALO, T.slot, bar);
        tma_load_3d(smem_u32(&P.S.dp), &M.m[6 + i], T.x0 - HALO, T.z0 - HALO, T.slot, bar);
    }
    __device__ __forceinline__ void prefetch(const FlowItem &, int) const {}
    __device__ __forceinline__ void fill(const FlowItem &it) const {
        copy_item<RJ>(P.k, A.c.kap, A.c, it.T, tid);
        copy_item<RJ>(P.dk, A.dkap, A.c, it.T, tid);
    }
    __device__ __forceinline__ void begin(const FlowItem &) const {}
    __device__ __forceinline__ void open(const FlowItem &) const {}
    __device__ __forceinline__ void close(const FlowItem &) const {}
    template <class MidFn>
    __device__ __forceinline__ void body(const FlowItem &it, const TileEdge &We, MidFn mid) const {
        if (it.T.flags & TI_FULL2) joint_tile<true>(A, P, We, it, tid, mid);
        else joint_tile<false>(A, P, We, it, tid, mid);
    }
};

__global__ void __launch_bounds__(NTJ, 1)
    born_joint_kernel(const __grid_constant__ BornFlow A, const __grid_constant__ TileMaps M) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    JointSmem &P = *reinterpret_cast<JointSmem *>(smem_raw);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_flow<kJointStageBytes, NCOREJ, LEADERJ>(A.f, A.c, PairLoopSmem{&P.S, P.We, &P.tail}, tid,
                                                JointK{A, M, P, tid});
}

// ---------------------------------------------------------------------------
// Two-step adjoint: steps k (nu^{k+1} -> nu^k) and k-1, the layout of
// fwd_pair_kernel.  The data of step k are added to the staged D_nu (D' = D +
// kappa r^{k-1}, ring included), those of step k-1 to the core's D_nu^k after
// step k.  The image accumulator takes a^{k-1} nu^k (tiles whose record reaches
// step k) and then a^{k-2} nu^{k-1}, in that order, as two one-step launches
// would.  Item arrays: nu^{k-1}, D_nu^{k-1}, image, a^{k-1}, a^{k-2}.
// ---------------------------------------------------------------------------
template <bool FULL, class MidFn>
__device__ __forceinline__ void adj_pair_tile(const AdjFlow &A, Pair2Stage &S, VTile &V, ItemSlots &I,
                                              const TileEdge &We, const FlowItem &it, int tid, MidFn mid) {
    const TileInfo &T = it.T;
    int lx, lz;
    item_of<R4>(tid, lx, lz);
    const bool core = tid < NCORE;
    const int nrow = FULL ? R4 : A.c.NZ - (T.z0 + lz);
    const bool ok = core && (FULL || T.x0 + lx < T.nxw);
    const int off = lz * T.pitch + lx;

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
    const bool image_k = T.nt > it.n - 1;
    q4 gq{}, a1q{}, a2q{};
    auto fetch = [&](int rr) {
        if (ok && rr < nrow) {
            const int o = off + rr * T.pitch;
            gq = ld4(it.p[2] + o);
            if (image_k) a1q = ld4(it.p[3] + o);
            a2q = ld4(it.p[4] + o);
        }
    };
    fetch(0);
    __syncthreads();  // nu^k and D_nu^k complete; the stage is no longer read
    // Data of step k-1 at the tile's receivers: D' = D_nu^k + kappa r^{k-2}.
    if (T.rec_end > T.rec_begin) {
        const float *rk = it.row - T.nrec;
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
            const int o = off + rr * T.pitch;
            st4(it.p[1] + o, d2);
            st4(it.p[0] + o, nn);
            st4(it.p[2] + o, g);
        }
    }
}

struct AdjK {
    const AdjFlow &A;
    const TileMaps &M;
    const PairSmem<ItemSlots> &P;
    InjBuf &IB;
    int tid;
    __device__ __forceinline__ int step(int m) const { return A.k1 - 2 * m; }
    __device__ __forceinline__ int count(int m) const { return active_count(A.f, step(m) - 2); }
    // Pairs of this launch before m in which the shot was active (nt > k - 2).
    __device__ __forceinline__ int need(int m, const TileInfo &T) const {
        const int x = A.k1 - 2 - T.nt;
        return x < 0 ? m : m - (x / 2 + 1);
    }
    __device__ __forceinline__ float *ptr(int i, int m, const TileInfo &T) const {
        const int k = step(m);
        const long long c = cell0(T);
        if (i < 2) return (i == 0 ? A.nu[(m + 1) & 1] : A.d[(m + 1) & 1]) + c;
        if (i == 2) return A.g + c;
        return i < 5 ? a_at(A.a, k - (i - 2)) + c : nullptr;
    }
    __device__ __forceinline__ float *row(int m, const TileInfo &T) const {
        return const_cast<float *>(A.r) + T.doff + (long long)(step(m) - 1) * T.nrec;
    }
    __device__ __forceinline__ void issue(const FlowItem &it, unsigned bar) const {
        const TileInfo &T = it.T;
        tma_load_3d(smem_u32(&P.S.u), &M.m[it.m & 1], T.x0 - HALO2, T.z0 - HALO2, T.slot, bar);
        tma_load_3d(smem_u32(&P.S.d), &M.m[2 + (it.m & 1)], T.x0 - HALO, T.z0 - HALO, T.slot, bar);
    }
    // The image and the a terms, which the second step loads from global memory.
    __device__ __forceinline__ void prefetch(const FlowItem &it, int lane) const {
        prefetch_rows(it.p[2], it.T, A.c.NZ, lane);
        if (it.T.nt > it.n - 1) prefetch_rows(it.p[3], it.T, A.c.NZ, lane);
        prefetch_rows(it.p[4], it.T, A.c.NZ, lane);
    }
    __device__ __forceinline__ void fill(const FlowItem &it) const { copy_item<R4>(P.I.k, A.c.kap, A.c, it.T, tid); }
    // Data of step k: the warp before the leader warp, free in the second step,
    // lists the next tile's grown-region injection (kappa and the receivers'
    // summed data, from global memory) while the core warps run that step;
    // after the tile's stage lands every thread adds the list to the staged
    // D_nu, D' = fmaf(kappa, sum, D).  A grown region with more receivers than
    // the list holds is injected from global memory then.  Shots whose record
    // ends before step k take none.
    __device__ __forceinline__ bool entry(const FlowItem &it, int e, int xb, int xe, InjEntry &en) const {
        if (e != xb && A.c.xrecs[e - 1].cell == A.c.xrecs[e].cell) return false;
        const TileInfo &T = it.T;
        const int cell = A.c.xrecs[e].cell, ez = cell / E, ex = cell % E;
        en.off = cell;
        en.kap = A.c.kap[(long long)T.mc * A.c.mstride + (long long)(T.z0 - HALO + ez) * A.c.pf + T.mx + ex - HALO];
        en.sum = receiver_sum(A.c.xrecs, e, xe, it.row);
        return true;
    }
    __device__ __forceinline__ void begin(const FlowItem &it) const {
        if (tid < LEADER2 - 32 || tid >= LEADER2) return;
        const int lane = tid & 31;
        const int xb = A.c.xrec_off[it.tile], xe = it.T.nt > it.n - 1 ? A.c.xrec_off[it.tile + 1] : xb;
        if (xe - xb <= kInjCap)
            for (int e = xb + lane; e < xe; e += 32) {
                InjEntry en{-1, 0.f, 0.f};
                entry(it, e, xb, xe, en);
                IB.e[e - xb] = en;
            }
        if (lane == 0) IB.n = xe - xb;
    }
    __device__ __forceinline__ void close(const FlowItem &it) const { begin(it); }
    __device__ __forceinline__ void open(const FlowItem &it) const {
        const int n = IB.n;  // uniform: written before the last barrier
        if (n == 0) return;
        float *dflat = &P.S.d[0][0];
        const int xb = A.c.xrec_off[it.tile];
        for (int e = tid; e < n; e += NT2) {
            InjEntry en{-1, 0.f, 0.f};
            if (n <= kInjCap) en = IB.e[e];
            else entry(it, xb + e, xb, xb + n, en);
            if (en.off >= 0) dflat[en.off] = fmaf(en.kap, en.sum, dflat[en.off]);
        }
        __syncthreads();
    }
    template <class MidFn>
    __device__ __forceinline__ void body(const FlowItem &it, const TileEdge &We, MidFn mid) const {
        if (it.T.flags & TI_INTERIOR2) adj_pair_tile<true>(A, P.S, P.V, P.I, We, it, tid, mid);
        else adj_pair_tile<false>(A, P.S, P.V, P.I, We, it, tid, mid);
    }
};

__global__ void __launch_bounds__(NT2, 2)
    adj_pair_kernel(const __grid_constant__ AdjFlow A, const __grid_constant__ TileMaps M) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PairSmem<ItemSlots> P(smem_raw);
    InjBuf &IB = *reinterpret_cast<InjBuf *>(smem_raw + kPair2Smem);
    const int tid = threadIdx.x + threadIdx.y * 32;
    run_flow<kPair2StageBytes, NCORE, LEADER2>(A.f, A.c, P.loop(), tid, AdjK{A, M, P, IB, tid});
}

// At most one CTA per tile.  Several pairs: a cooperative launch.  One pair: a
// programmatic dependent of the launch before.
template <typename K, typename Args>
void launch_flow(K kernel, size_t smem, int threads, int cap, const Args &a, const TileMaps &maps, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(a.f.nt, cap));
    cfg.blockDim = dim3(32, threads / 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (a.f.npairs > 1) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, a, maps);
}

// CTAs of a kernel that are resident at once on the current device.
template <auto KERNEL, size_t SMEM, int THREADS>
int resident() {
    static PerDevice ctas;
    int dev = 0;
    cudaGetDevice(&dev);
    return ctas.get(dev, [&] {
        int n = 0, sms = 1;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaFuncSetAttribute((const void *)KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, (const void *)KERNEL, THREADS, SMEM);
        return std::max(n, 1) * sms;
    });
}

int cap_fwd(int store) {
    return store == ST_A    ? resident<fwd_pair_kernel<ST_A>, kPair2Smem, NT2>()
           : store == ST_CK ? resident<fwd_pair_kernel<ST_CK>, kPair2Smem, NT2>()
                            : resident<fwd_pair_kernel<ST_NONE>, kPair2Smem, NT2>();
}
int cap_adj() { return resident<adj_pair_kernel, kAdj2Smem, NT2>(); }
int cap_born() { return resident<born_pair_kernel, kBorn2Smem, NT2>(); }
int cap_joint() { return resident<born_joint_kernel, sizeof(JointSmem), NTJ>(); }

}  // namespace

int flow_ctas(int kind) {
    switch (kind) {
    case FLOW_FWD: return std::min(cap_fwd(ST_A), std::min(cap_fwd(ST_CK), cap_fwd(ST_NONE)));
    case FLOW_ADJ: return cap_adj();
    case FLOW_BORN_HIST: return cap_born();
    default: return cap_joint();
    }
}

void launch_fwd_flow(const FwdFlow &a, const TileMaps &maps, cudaStream_t s) {
    if (a.a.base) launch_flow(fwd_pair_kernel<ST_A>, kPair2Smem, NT2, cap_fwd(ST_A), a, maps, s);
    else if (a.ck) launch_flow(fwd_pair_kernel<ST_CK>, kPair2Smem, NT2, cap_fwd(ST_CK), a, maps, s);
    else launch_flow(fwd_pair_kernel<ST_NONE>, kPair2Smem, NT2, cap_fwd(ST_NONE), a, maps, s);
}

void launch_adj_flow(const AdjFlow &a, const TileMaps &maps, cudaStream_t s) {
    launch_flow(adj_pair_kernel, kAdj2Smem, NT2, cap_adj(), a, maps, s);
}

void launch_born_hist_flow(const BornFlow &a, const TileMaps &maps, cudaStream_t s) {
    launch_flow(born_pair_kernel, kBorn2Smem, NT2, cap_born(), a, maps, s);
}

void launch_born_joint_flow(const BornFlow &a, const TileMaps &maps, cudaStream_t s) {
    launch_flow(born_joint_kernel, sizeof(JointSmem), NTJ, cap_joint(), a, maps, s);
}

}  // namespace dhfwi
