// resident.cuh -- small FP32 grids advanced T steps by one launch, the state
// held in the registers of one thread-block cluster.
//
// A run of a small grid through the temporal kernel is a chain of launches that
// each last a few microseconds, almost all of it latency: launch, load, a
// 2K-beat fill, store.  Here the grid's rows are dealt out once, in order, to
// the warps of a cluster (16 thread blocks of W warps); a warp keeps its
// NR = 1 .. 4 whole rows in registers, lane l holding columns V l .. V l + V - 1,
// and the planes are read once and written once per launch, each cell by the
// thread that holds it.  Per step a warp hands its first and last row to the
// warps above and below through shared memory, and waits for theirs on an
// mbarrier of its own: within a block plain stores and an arrival, across a
// block edge asynchronous stores into the other block's shared memory, whose
// bytes the mbarrier counts.  What needs no handed row (all shuffles, the inner
// rows) is done before the wait.
//
// Columns: west and east neighbours across lanes are shuffles around the ring of
// the lanes in use, so a row wraps (or ends, under zero flux) inside its warp.
// A width that is no multiple of V gives the last lane in use the last V
// columns, overlapping the lane before it (RAG): the columns held twice are
// computed twice, with the same bits, and only the two shuffles between these
// lanes take another element (Ring).
//
// Every cell is formed by nbr_sum's grouping and cell_react: the bits of the
// other variants.  On the torus the pair sums (n + w), (s + e) are formed once
// and used by two rows, as in temporal.cuh.
//
// Handed rows have two slots, by step parity.  A slot is written for step t + 2
// by a neighbour that has the receiver's row of step t + 1, which was formed from
// the slot's row of step t: the slot has been read, and its mbarrier's phase of
// step t is over.  Each row handed on is waited for by its receiver, and the
// blocks leave together, so none is written after its block has left.
//
// Waits are bounded.  A warp whose wait gives up sets a flag in every block and
// ends (give_up): it hands on no more rows, so its neighbours' waits give up in
// turn.  The flag is read after the barrier that ends the steps, and every warp
// of the cluster then stores NaNs in both planes, over its rows: a failed run has
// no cell that looks like a result.
//
// Bound: latency of the hand-over up to 128^2 (64^2: 345 cycles a step, of which
// about 100 are the sums and the update), one warp's issue rate per scheduler of
// 16 SMs at 256^2.  us a step, launches -> resident: 64^2 0.84 -> 0.17, 128^2 0.82
// -> 0.23, 256^2 0.86 -> 0.47.  Measured on the way, 64^2 / 128^2 / 256^2: one
// cluster barrier a step 0.34 / 0.46 / 0.68; every row by asynchronous stores
// 0.26 / 0.38 / 0.74; two rows handed on every second step, with the redundant
// rows computed, 0.21 / 0.29 / 0.71.
#pragma once

#include "common.cuh"

namespace rdk {

constexpr int kResRows = 4;  // most rows of a warp

struct ResArgs {
    float *u, *v;  // state planes, in place
    int nn, nm, steps, blocks, warps;  // blocks of the cluster, warps of a block
    Coef<float> p;
    uint64_t wait_ns;  // limit of a wait
    int never;         // arrivals that no warp makes: 1 has every wait give up (for tests)
};

// Most warps of a block: V = 12 needs up to 255 registers a thread, V = 8 up to
// 225, V = 4 up to 127, V = 2 up to 96.
template <int V> struct ResWarps : IntC<V >= 8 ? 8 : 16> {};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// A shared-memory address of this block as the same address of block `rank`.
__device__ __forceinline__ unsigned in_cluster(unsigned a, unsigned rank) {
    unsigned q;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(q) : "r"(a), "r"(rank));
    return q;
}

// The lanes of a row as a ring: lane `last` is the last one in use.  With RAG
// it holds the last V columns, the first V - rem of them also held by the lane
// before it (rem = NM mod V): its west neighbour is that lane's element rem - 1,
// and that lane's east neighbour is its element V - rem.
// RAG = 1: any width; 4: widths that are multiples of 4, so that rem is one and
// fewer elements are to choose from (V = 12; with V = 8 it made no difference).
template <int V, int BC, int RAG> struct Ring {
    int west_src, east_src;
    bool first, end;         // lane holds column 0 / the last column
    bool pw[V], pe[V];       // element handed west -> east / east -> west by this lane
    __device__ __forceinline__ Ring(int lane, int last, int rem) {
        first = (lane == 0);
        end = (lane == last);
        west_src = first ? last : lane - 1;
        east_src = lane >= last ? 0 : lane + 1;
#pragma unroll
        for (int k = 0; k < V; ++k) {
            pw[k] = RAG > 0 && lane == last - 1 && k == rem - 1;
            pe[k] = RAG > 0 && end && k == V - rem;
        }
    }
    // Element -1 of a row held as a[0 .. V-1] by the lanes.
    __device__ __forceinline__ float west(const float (&a)[V]) const {
        float x = a[V - 1];
        if constexpr (RAG > 0) {
#pragma unroll
            for (int k = RAG - 1; k < V - 1; k += RAG) x = pw[k] ? a[k] : x;
        }
        x = __shfl_sync(kFull, x, west_src);
        return (BC == BC_MIRROR && first) ? a[0] : x;
    }
    // Element V.
    __device__ __forceinline__ float east(const float (&a)[V]) const {
        float x = a[0];
        if constexpr (RAG > 0) {
#pragma unroll
            for (int k = RAG; k < V; k += RAG) x = pe[k] ? a[k] : x;
        }
        x = __shfl_sync(kFull, x, east_src);
        return (BC == BC_MIRROR && end) ? a[V - 1] : x;
    }
};

// A lane's V values of a handed row: 16-byte (V = 2: 8-byte) accesses, lanes
// consecutive.  Within the block a plain store, whose sender then arrives at
// the receiving warp's mbarrier; to another block an asynchronous store (`a`
// and `bar` are cluster-window addresses), whose bytes that mbarrier counts.
template <int V>
__device__ __forceinline__ void hand_store(unsigned a, const float (&x)[V]) {
    if constexpr (V == 2) {
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x[0]), "f"(x[1]) : "memory");
    } else {
#pragma unroll
        for (int c = 0; c < V; c += 4)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a + c * 128), "f"(x[c]), "f"(x[c + 1]),
                         "f"(x[c + 2]), "f"(x[c + 3])
                         : "memory");
    }
}
template <int V>
__device__ __forceinline__ void hand_store_far(unsigned a, unsigned bar, const float (&x)[V]) {
    if constexpr (V == 2) {
        asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(a),
                     "f"(x[0]), "f"(x[1]), "r"(bar)
                     : "memory");
    } else {
#pragma unroll
        for (int c = 0; c < V; c += 4)
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                             a + c * 128),
                         "f"(x[c]), "f"(x[c + 1]), "f"(x[c + 2]), "f"(x[c + 3]), "r"(bar)
                         : "memory");
    }
}

// The warp's mbarriers, one per step parity: a phase takes the arrivals of the
// neighbours in the block, and for rows from other blocks the warp's own
// arrival, which states their bytes, and those bytes.
__device__ __forceinline__ void bar_init(unsigned bar, unsigned arrivals) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(arrivals) : "memory");
}
// The arrivals of the threads with p (one lane of a warp): predicated, so that
// the warp does not branch.
__device__ __forceinline__ void bar_arrive(bool p, unsigned bar) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %1, 0;\n@q mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n}" ::"r"(bar),
                 "r"((unsigned)p)
                 : "memory");
}
__device__ __forceinline__ void bar_expect(bool p, unsigned bar, unsigned bytes) {
    asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\n@q mbarrier.arrive.expect_tx.relaxed.cta.shared::cta.b64 _, [%0], %1;\n}" ::"r"(bar),
                 "r"(bytes), "r"((unsigned)p)
                 : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t clock_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// False when the phase has not completed for `limit` ns.  The blocks of a cluster
// run at the same time, so with the usual limit only a fault of this file could
// do that.
constexpr uint64_t kResWaitNs = 10ull * 1000 * 1000 * 1000;
constexpr uint64_t kResGiveUpNs = 1000 * 1000;  // where the wait is meant to run out
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned parity, uint64_t limit) {  // the whole warp, with one answer
    bool ok = bar_try(bar, parity);
    if (__all_sync(kFull, ok)) return true;
    const uint64_t t0 = clock_ns();
    for (;;) {
        ok = ok || bar_try(bar, parity);
        if (__all_sync(kFull, ok)) return true;
        if (__any_sync(kFull, clock_ns() - t0 > limit)) return false;
    }
}
// The cluster's failure flag: a word behind the mbarriers of each block.
constexpr uint64_t kResDrainNs = 1000 * 1000;  // an asynchronous store takes about a microsecond
__device__ __forceinline__ void flag_set(unsigned flag, unsigned rank) {  // block `rank`'s
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(in_cluster(flag, rank)), "r"(1u) : "memory");
}
__device__ __forceinline__ bool flag_get(unsigned flag) {
    unsigned x;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x) : "r"(flag) : "memory");
    return x != 0;
}
// After a failure: NaNs in the warp's rows, over what it has stored.  Handed rows that
// nobody waited for may still be on their way: no block leaves before they are in.
__device__ __forceinline__ void spoil(const ResArgs &a, int r0, int nr) {
    __syncwarp();
#pragma unroll 1
    for (int i = threadIdx.x & 31; i < nr * a.nm; i += 32)
        a.u[(int64_t)r0 * a.nm + i] = a.v[(int64_t)r0 * a.nm + i] = __int_as_float(0x7fffffff);
    const uint64_t t0 = clock_ns();
    while (!__any_sync(kFull, clock_ns() - t0 >= kResDrainNs)) {}
    cluster_arrive();
    cluster_wait();
}
// The end of a warp (rows r0 .. r0 + nr - 1) whose wait gave up: the barriers that
// the others pass after their last step, and the thread's exit.  The exit has a
// predicate (always true: a cluster has blocks), so that the compiler sees no way
// out of the step loop here; with one, it builds the loop otherwise: us a step at
// 64^2 / 128^2 / 256^2, a flag and a break 0.196 / 0.265 / 0.476, an exit known as
// such 0.188 / 0.255 / 0.508, this 0.167 / 0.232 / 0.470.
__device__ __forceinline__ void give_up(const ResArgs &a, int r0, int nr, unsigned flag) {
    const int lane = threadIdx.x & 31;
    if (lane < a.blocks) flag_set(flag, lane);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    spoil(a, r0, nr);
    asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %0, 0;\n@q exit;\n}" ::"r"(a.blocks) : "memory");
}
template <int V>
__device__ __forceinline__ void hand_load(unsigned a, float (&x)[V]) {
    if constexpr (V == 2) {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x[0]), "=f"(x[1]) : "r"(a) : "memory");
    } else {
#pragma unroll
        for (int c = 0; c < V; c += 4)
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(x[c]), "=f"(x[c + 1]), "=f"(x[c + 2]), "=f"(x[c + 3])
                         : "r"(a + c * 128)
                         : "memory");
    }
}

__device__ __forceinline__ float hand_load1(unsigned a) {
    float x;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
    return x;
}

template <int V>
__device__ __forceinline__ void copy_row(float (&d)[V], const float (&s)[V]) {
#pragma unroll
    for (int e = 0; e < V; ++e) d[e] = s[e];
}

// One field of the warp's rows over a step: the neighbour sums, each row's once.
// e[q], w[q]: elements V and -1 of row q.
// Torus: pair(q)(j) = row_{q-1}(j+1) + row_q(j), and the sum of cell (q, j) is
// pair(q)(j-1) + pair(q+1)(j).  pair(q)(-1) = row_{q-1}(0) + row_q(-1) is formed
// from the row's own shuffle, so that no shuffle waits for another.
// Zero flux: (n + s) + (w + e).
template <int V, int NR, int BC> struct RowSums {
    float e[NR], w[NR];
    float keep[V], keep_w;    // torus: pair(1); zero flux: row 1, both for row 0's sum
    float above[V], above_w;  // torus: pair(q); zero flux: row q - 1

    template <class RING>
    __device__ __forceinline__ void shuffles(const RING &r, const float (&x)[NR][V]) {
#pragma unroll
        for (int q = 0; q < NR; ++q) {
            e[q] = r.east(x[q]);
            w[q] = r.west(x[q]);
        }
    }
    // pair of the rows n (its element V: ne) above c (its element -1: cw).
    static __device__ __forceinline__ void pair(const float (&n)[V], float ne, const float (&c)[V], float cw,
                                                float (&o)[V], float &ow) {
#pragma unroll
        for (int j = 0; j < V; ++j) o[j] = add_rn(j == V - 1 ? ne : n[j + 1], c[j]);
        ow = add_rn(n[0], cw);
    }
    static __device__ __forceinline__ void join(const float (&a)[V], float aw, const float (&b)[V], float (&s)[V]) {
#pragma unroll
        for (int j = 0; j < V; ++j) s[j] = add_rn(j == 0 ? aw : a[j - 1], b[j]);
    }
    static __device__ __forceinline__ void plain(const float (&n)[V], const float (&c)[V], const float (&s)[V], float cw,
                                                 float ce, float (&o)[V]) {
#pragma unroll
        for (int j = 0; j < V; ++j)
            o[j] = nbr_sum<BC>(n[j], s[j], j == 0 ? cw : c[j - 1], j == V - 1 ? ce : c[j + 1]);
    }

    // Two or more rows, ready for row 1.
    __device__ __forceinline__ void start(const float (&x0)[V], const float (&x1)[V]) {
        if constexpr (BC == BC_WRAP) {
            pair(x0, e[0], x1, w[NR > 1 ? 1 : 0], keep, keep_w);
            copy_row(above, keep);
            above_w = keep_w;
        } else {
            copy_row(keep, x1);
            copy_row(above, x0);
        }
    }
    // Sum of row q (c), row q + 1 (s) below it; then ready for row q + 1.
    __device__ __forceinline__ void next(int q, const float (&c)[V], const float (&s)[V], float (&o)[V]) {
        if constexpr (BC == BC_WRAP) {
            float nx[V], nw;
            pair(c, e[q], s, q + 1 < NR ? w[q + 1 < NR ? q + 1 : 0] : 0.0f, nx, nw);  // nw of the last row is not used
            join(above, above_w, nx, o);
            copy_row(above, nx);
            above_w = nw;
        } else {
            plain(above, c, s, w[q], e[q], o);
            copy_row(above, c);
        }
    }
    // Sum of row 0 (c) below the handed row n (its element V: ne), after start().
    __device__ __forceinline__ void top(const float (&n)[V], float ne, const float (&c)[V], float (&o)[V]) {
        if constexpr (BC == BC_WRAP) {
            float p[V], pw;
            pair(n, ne, c, w[0], p, pw);
            join(p, pw, keep, o);
        } else {
            plain(n, c, keep, w[0], e[0], o);
        }
    }
    // Sum of a warp's only row between the handed rows n and s.
    __device__ __forceinline__ void only(const float (&n)[V], float ne, const float (&c)[V], const float (&s)[V],
                                         float (&o)[V]) {
        if constexpr (BC == BC_WRAP) {
            float p[V], pw, nx[V], nw;
            pair(n, ne, c, w[0], p, pw);
            pair(c, e[0], s, 0.0f, nx, nw);
            join(p, pw, nx, o);
        } else {
            plain(n, c, s, w[0], e[0], o);
        }
    }
};

// The whole run of a warp that holds NR rows from row r0 on; w = its index in
// the block, g = in the cluster.
template <int V, int NR, int RX, int BC, int RAG>
__device__ __forceinline__ void resident_rows(const ResArgs &a, int r0, int w, int g, unsigned rank, unsigned smem) {
    constexpr bool OUT = (RX == RX_CENN);   // sums over the outputs clamp1(u); v is constant
    constexpr int F = OUT ? 1 : 2;          // handed fields
    const int lane = threadIdx.x & 31;
    const int last = (a.nm - 1) / V;
    const Ring<V, BC, RAG> ring(lane, last, a.nm % V);
    const int col = RAG > 0 && lane == last ? a.nm - V : lane * V;
    const bool in_use = lane <= last;

    float U[NR][V], W[NR][V];
#pragma unroll
    for (int q = 0; q < NR; ++q)
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const int64_t off = (int64_t)(r0 + q) * a.nm + col + e;
            U[q][e] = in_use ? a.u[off] : 0.0f;
            W[q][e] = in_use ? a.v[off] : 0.0f;
        }

    // slot (parity, warp, direction, field): direction 0 = the row above the
    // warp's first, 1 = the row below its last
    constexpr unsigned kSlot = 128 * V;
    const unsigned buf_step = a.warps * 2 * F * kSlot;
    auto slot = [&](int warp, int dir, int ln) {
        return smem + (warp * 2 + dir) * F * kSlot + ln * (V == 2 ? 8 : 16);
    };
    const bool up_far = w == 0 && a.blocks > 1, down_far = w == a.warps - 1 && a.blocks > 1;
    const int nwarps = a.blocks * a.warps;
    const bool top = (BC == BC_MIRROR) && g == 0, bottom = (BC == BC_MIRROR) && g == nwarps - 1;
    // where the first / last row and their arrivals go (parity 0)
    const unsigned bars = smem + 2 * buf_step;  // [warp][parity]
    const unsigned bar = bars + 16 * w, flag = bars + 16 * a.warps;
    const int up_w = w == 0 ? a.warps - 1 : w - 1, down_w = w == a.warps - 1 ? 0 : w + 1;
    const unsigned up_rank = rank == 0 ? a.blocks - 1 : rank - 1;
    const unsigned down_rank = (int)rank == a.blocks - 1 ? 0 : rank + 1;
    unsigned up_to = slot(up_w, 1, lane), up_bar = bars + 16 * up_w;
    unsigned down_to = slot(down_w, 0, lane), down_bar = bars + 16 * down_w;
    if (up_far) up_to = in_cluster(up_to, up_rank), up_bar = in_cluster(up_bar, up_rank);
    if (down_far) down_to = in_cluster(down_to, down_rank), down_bar = in_cluster(down_bar, down_rank);
    const unsigned from = slot(w, 0, lane);
    // element V of the handed row above, where its lane stored it
    const int east_e = RAG > 0 && lane == last - 1 ? V - a.nm % V : 0;
    const unsigned from_east = slot(w, 0, ring.east_src) + (east_e / 4) * 512 + (east_e % 4) * 4;
    // bytes from the neighbours in other blocks
    const unsigned bytes = ((int)(up_far && !top) + (int)(down_far && !bottom)) * F * kSlot;
    // lane 0's arrivals: at the neighbours in this block, and for those bytes
    const bool tell_up = lane == 0 && !top && !up_far, tell_down = lane == 0 && !bottom && !down_far;
    const bool expect = lane == 0 && bytes > 0;
    const bool alone = top && bottom;  // nobody hands this warp a row
    float Y[OUT ? NR : 1][V];
    float su[V], sv[V];
    auto react = [&](int q) {
#pragma unroll
        for (int e = 0; e < V; ++e)
            cell_react<float, RX>(U[q][e], W[q][e], su[e], OUT ? 0.0f : sv[e], OUT ? Y[OUT ? q : 0][e] : 0.0f, a.p, U[q][e],
                                  W[q][e]);
    };
    auto &X = [&]() -> float(&)[NR][V] {  // what the first field's sums run over
        if constexpr (OUT) return Y;
        else return U;
    }();
    auto hand = [&](int q, unsigned to, unsigned to_bar, bool far) {
        if (far) {
            hand_store_far<V>(to, to_bar, X[q]);
            if constexpr (!OUT) hand_store_far<V>(to + kSlot, to_bar, W[q]);
        } else {
            hand_store<V>(to, X[q]);
            if constexpr (!OUT) hand_store<V>(to + kSlot, W[q]);
        }
    };

    for (int t = 0; t < a.steps; ++t) {
        const int b = t & 1;
        if constexpr (OUT) {
#pragma unroll
            for (int q = 0; q < NR; ++q)
#pragma unroll
                for (int e = 0; e < V; ++e) Y[q][e] = clamp1(U[q][e]);
        }
        if (!top) hand(0, up_to + b * buf_step, up_bar + 8 * b, up_far);
        if (!bottom) hand(NR - 1, down_to + b * buf_step, down_bar + 8 * b, down_far);
        __syncwarp();
        bar_arrive(tell_up, up_bar + 8 * b);
        bar_arrive(tell_down, down_bar + 8 * b);
        bar_expect(expect, bar + 8 * b, bytes);
        // what needs no handed row
        RowSums<V, NR, BC> qu, qv;
        qu.shuffles(ring, X);
        if constexpr (!OUT) qv.shuffles(ring, W);
        if constexpr (NR >= 2) {
            qu.start(X[0], X[1]);
            if constexpr (!OUT) qv.start(W[0], W[1]);
#pragma unroll
            for (int q = 1; q < NR - 1; ++q) {
                qu.next(q, X[q], X[q + 1], su);
                if constexpr (!OUT) qv.next(q, W[q], W[q + 1], sv);
                react(q);
            }
        }
        if (!alone && !bar_wait(bar + 8 * b, (t >> 1) & 1, a.wait_ns)) give_up(a, r0, NR, flag);
        float nu[V], nv[V], bu[V], bv[V], nue = 0.0f, nve = 0.0f;  // the handed rows above and below
        const unsigned at = from + b * buf_step;
        hand_load<V>(at, nu);
        hand_load<V>(at + F * kSlot, bu);
        if constexpr (BC == BC_WRAP) nue = hand_load1(from_east + b * buf_step);
        if constexpr (!OUT) {
            hand_load<V>(at + kSlot, nv);
            hand_load<V>(at + F * kSlot + kSlot, bv);
            if constexpr (BC == BC_WRAP) nve = hand_load1(from_east + b * buf_step + kSlot);
        }
        if (BC == BC_MIRROR) {  // beyond an edge: the edge row itself
#pragma unroll
            for (int e = 0; e < V; ++e) {
                nu[e] = top ? X[0][e] : nu[e];
                bu[e] = bottom ? X[NR - 1][e] : bu[e];
                if constexpr (!OUT) {
                    nv[e] = top ? W[0][e] : nv[e];
                    bv[e] = bottom ? W[NR - 1][e] : bv[e];
                }
            }
        }
        if constexpr (NR == 1) {
            qu.only(nu, nue, X[0], bu, su);
            if constexpr (!OUT) qv.only(nv, nve, W[0], bv, sv);
            react(0);
        } else {
            qu.next(NR - 1, X[NR - 1], bu, su);
            if constexpr (!OUT) qv.next(NR - 1, W[NR - 1], bv, sv);
            react(NR - 1);
            qu.top(nu, nue, X[0], su);
            if constexpr (!OUT) qv.top(nv, nve, W[0], sv);
            react(0);
        }
    }

    if (in_use) {
#pragma unroll
        for (int q = 0; q < NR; ++q)
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const int64_t off = (int64_t)(r0 + q) * a.nm + col + e;
                a.u[off] = U[q][e];
                if constexpr (!OUT) a.v[off] = W[q][e];
            }
    }
    // every warp has done its steps or given up: nothing is handed on from here
    cluster_arrive();
    cluster_wait();
    if (flag_get(flag)) spoil(a, r0, NR);  // the same answer in the whole cluster
}

// One cluster; warp g of it holds rows g NN / nwarps .. (g + 1) NN / nwarps - 1.
template <int V, int RX, int BC, int RAG>
__global__ void __launch_bounds__(32 * ResWarps<V>::value, 1)
k_resident(const ResArgs a) {
    extern __shared__ __align__(16) unsigned char res_smem[];
    pdl_wait();
    unsigned rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const unsigned smem = (unsigned)__cvta_generic_to_shared(res_smem);
    const int w = threadIdx.x >> 5;
    const int g = (int)rank * a.warps + w;
    const int nwarps = a.blocks * a.warps;
    const int r0 = (int)((int64_t)g * a.nn / nwarps);
    const int nr = (int)((int64_t)(g + 1) * a.nn / nwarps) - r0;
    if ((threadIdx.x & 31) == 0) {
        const unsigned bar = smem + 2 * a.warps * 2 * (RX == RX_CENN ? 1 : 2) * 128 * V + 16 * w;
        // arrivals: of the neighbours in this block, and one for the bytes from others
        const bool top = BC == BC_MIRROR && g == 0, bottom = BC == BC_MIRROR && g == nwarps - 1;
        const bool up_far = w == 0 && a.blocks > 1, down_far = w == a.warps - 1 && a.blocks > 1;
        const int n = (!top && !up_far) + (!bottom && !down_far) + ((!top && up_far) || (!bottom && down_far));
        bar_init(bar, max(n, 1) + a.never);
        bar_init(bar + 8, max(n, 1) + a.never);
        if (w == 0) asm volatile("st.shared.u32 [%0], %1;" ::"r"(bar + 16 * a.warps), "r"(0u) : "memory");  // no failure
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // every block's mbarriers and flag stand before another hands it a row
    cluster_arrive();
    cluster_wait();
    switch (nr) {  // 1 .. kResRows, chosen by the launcher
        case 1: resident_rows<V, 1, RX, BC, RAG>(a, r0, w, g, rank, smem); break;
        case 2: resident_rows<V, 2, RX, BC, RAG>(a, r0, w, g, rank, smem); break;
        case 3: resident_rows<V, 3, RX, BC, RAG>(a, r0, w, g, rank, smem); break;
        default: resident_rows<V, 4, RX, BC, RAG>(a, r0, w, g, rank, smem); break;
    }
    pdl_trigger();
}

}  // namespace rdk
