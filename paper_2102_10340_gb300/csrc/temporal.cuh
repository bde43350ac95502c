// temporal.cuh -- the K-step register pipeline shared by the single-grid and
// batched temporally blocked kernels (Eq. 1 applied K times per HBM pass).
//
// A warp owns one (band, strip) work item: output columns
// [band*OUTW, band*OUTW + OUTW) and output rows [strip*rows, strip*rows + rows)
// of an NN x NM torus.  It loads 32*V columns starting H*V columns to the left
// of its band (H = ceil(K/V) halo lanes per side, indices wrapped modulo NM)
// and input rows r0-K .. r0+rows+K-1 (wrapped modulo NN).  Input rows are
// staged through a per-warp shared-memory ring by cp.async, two or three rows
// ahead of use.  Each input row passes through K stages held in registers;
// stage s turns rows (q-1, q, q+1)
// of stage s-1 into row q of stage s.  After K stages the K outermost columns
// on each side are stale, which is why only lanes H .. 31-H store.
//
// Zero-flux boundary (BC_MIRROR): the halo rows and columns beyond a grid
// edge are loaded as the mirror image of the rows and columns inside it
// (row -1 <- row 0, row -2 <- row 1, ...; a lane whose 16-byte vector lies
// beyond an edge loads the mirrored vector and reverses its elements).  The
// 2N x 2M torus holding that mirror image evolves exactly like the zero-flux
// grid (the edge faces are mirror planes and the update keeps a mirrored
// state mirrored), so every stage sees the edge cell as its own outside
// neighbour with no per-stage test; only the input indexing differs.  Sums
// of mirrored pairs are formed in swapped order, which IEEE addition does not
// notice: the results are the bits the single-step kernel computes.
//
// Ragged rows (T = Ragged<E>: NM no multiple of the lane width, or planes off
// their 16-byte alignment): the same pipeline, with the band's elements
// copied one by one to their wrapped or reflected columns (coalesced: lane l
// copies elements l, l + 32, ...), read back as lane vectors, and stored one
// by one.  1003 x 1021, 100 steps: 224 us, against 758 with k_generic.
#pragma once

#include "common.cuh"

namespace rdk {

// Warps per block of every kernel built on temporal_strip.  One: the same
// resident warps per SM issue faster as one-warp blocks (K = 8 at 4096^2:
// 1436 against 1278 Gcell-updates/s with four-warp blocks and 1270 with
// two; ncu shows the dispatch stalls per issued instruction falling from
// 0.44 to 0.18 and issue-active rising from 63 % to 72 % at the same 8
// warps per SM and the same instructions).
constexpr int kTemporalWarps = 1;
// Input rows staged per warp by the three-phase pipelines (prefetch distance
// kRing - 1 = 2 beats, about 1.5 us of the K = 8 pipeline, above the HBM
// latency).  Three slots match the 3-beat window rotation, so a beat's slots
// are compile-time constants.  The two-phase pipelines keep kRing2 rows (a
// power of two; the slot of a beat is a running index).
constexpr int kRing = 3;
constexpr int kRing2 = 4;

// Per-lane 16-byte asynchronous global -> shared copy (cp.async, L2 only).
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
// 8-byte variant (16-bit storage: 4 values per lane); cp.async.cg takes 16 only.
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
// One element of an unaligned row (4 or 8 bytes).
template <int BYTES>
__device__ __forceinline__ void cp_async_elem(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Geometry of one (band, strip) work item for depth K and halo H.
// Input-row index q in 0 .. nout + 2K - 1 is global row r0 - K + q (wrapped,
// or reflected under zero flux); the strip owns rows q in [K, K + nout) and
// lanes H .. 31-H whose column sc = c0 + (lane - H) V is below NM.  lc is the
// first column the lane loads; rev marks a mirrored (reversed) vector.
// Ragged rows: the lane copies band positions lane + 32 e (consecutive lanes
// take consecutive elements), which are columns col[e]; nel of its own
// columns are below NM.
struct StripGeom {
    int lc, sc, r0, nout, total;
    bool st_lane, rev;
    int col[4], nel;
};

// Shared-memory ring of one warp: rows x {u, v} x 32 lanes x 16 bytes.
// Each lane copies and later reads back only its own 16 bytes, so the lane's
// own cp.async.wait_group is the only synchronisation needed; except in
// ragged rows, where a lane copies other elements than it reads back and the
// warp synchronises before both (ring_issue_at, ring_read_at).
template <typename T> struct RowRing {
    typedef typename Vec<T>::type VT;
    VT (*slot)[2][32];  // [row][field][lane]
};

template <typename T>
__device__ __forceinline__ void ring_issue_at(const RowRing<T> &r, int slot, int g, int nm, const StripGeom &geo,
                                              const T *__restrict__ u, const T *__restrict__ v) {
    const int lane = threadIdx.x & 31;
    if constexpr (IsRagged<T>::value) {
        __syncwarp();  // the slot has been read by every lane
        T *su = reinterpret_cast<T *>(&r.slot[slot][0][0]);
        T *sv = reinterpret_cast<T *>(&r.slot[slot][1][0]);
        const T *ru = u + (int64_t)g * nm;
        const T *rv = v + (int64_t)g * nm;
#pragma unroll
        for (int e = 0; e < Vec<T>::N; ++e) {
            cp_async_elem<sizeof(T)>(su + lane + 32 * e, ru + geo.col[e]);
            cp_async_elem<sizeof(T)>(sv + lane + 32 * e, rv + geo.col[e]);
        }
        return;
    }
    const int64_t off = (int64_t)g * nm + geo.lc;
    if constexpr (sizeof(typename Vec<T>::type) == 32) {  // two 16-byte halves per field
        char *su = reinterpret_cast<char *>(&r.slot[slot][0][lane]);
        char *sv = reinterpret_cast<char *>(&r.slot[slot][1][lane]);
        cp_async16(su, u + off);
        cp_async16(su + 16, reinterpret_cast<const char *>(u + off) + 16);
        cp_async16(sv, v + off);
        cp_async16(sv + 16, reinterpret_cast<const char *>(v + off) + 16);
    } else if constexpr (sizeof(typename Vec<T>::type) == 16) {
        cp_async16(&r.slot[slot][0][lane], u + off);
        cp_async16(&r.slot[slot][1][lane], v + off);
    } else {
        cp_async8(&r.slot[slot][0][lane], u + off);
        cp_async8(&r.slot[slot][1][lane], v + off);
    }
}

// Input row m goes to slot m % kRing.
template <typename T>
__device__ __forceinline__ void ring_issue(const RowRing<T> &r, int m, int g, int nm, const StripGeom &geo,
                                           const T *__restrict__ u, const T *__restrict__ v) {
    ring_issue_at(r, m % kRing, g, nm, geo, u, v);
}

template <typename T>
__device__ __forceinline__ void ring_read_at(const RowRing<T> &r, int slot, Slice<CT<T>, Vec<T>::N> &s) {
    typedef typename Vec<T>::type VT;
    const int lane = threadIdx.x & 31;
    if constexpr (IsRagged<T>::value) __syncwarp();  // every lane's copies have landed
    const VT a = r.slot[slot][0][lane];
    const VT b = r.slot[slot][1][lane];
    typedef typename std::conditional<IsRagged<T>::value, typename Base16<T>::type, T>::type E;
    unpack_vec<E, Vec<T>::N>(a, s.u);
    unpack_vec<E, Vec<T>::N>(b, s.v);
}

template <typename T>
__device__ __forceinline__ void ring_read(const RowRing<T> &r, int m, Slice<CT<T>, Vec<T>::N> &s) {
    ring_read_at(r, m % kRing, s);
}

// ring_read for boundary BC; under BC_MIRROR a lane whose columns lie beyond
// an edge (rev) reverses the element order of the mirrored vector it loaded.
template <typename T, int BC>
__device__ __forceinline__ void ring_read_bc(const RowRing<T> &r, int slot, bool rev, Slice<CT<T>, Vec<T>::N> &s) {
    ring_read_at(r, slot, s);
    if constexpr (BC == BC_MIRROR) {
        constexpr int V = Vec<T>::N;
        Slice<CT<T>, Vec<T>::N> t = s;
#pragma unroll
        for (int e = 0; e < V; ++e) {
            s.u[e] = rev ? t.u[V - 1 - e] : t.u[e];
            s.v[e] = rev ? t.v[V - 1 - e] : t.v[e];
        }
    }
}

// Source row of the strip's input rows, advanced one row per beat: wrapped
// on the torus; under zero flux the reflected sequence (..., 1, 0, 0, 1, ...
// at the top edge, ..., n-2, n-1, n-1, n-2, ... at the bottom).
template <int BC> struct RowWalk {
    int g = 0, dir = 1;
    __device__ __forceinline__ void start(int64_t r, int n) {
        if constexpr (BC == BC_MIRROR) {
            const int q = wrap_row(r, 2 * (int64_t)n);
            g = q < n ? q : 2 * n - 1 - q;
            dir = q < n ? 1 : -1;
        } else {
            g = wrap_row(r, n);
        }
    }
    __device__ __forceinline__ void next(int n) {
        if constexpr (BC == BC_MIRROR) {
            if (dir > 0) {
                if (g == n - 1) dir = -1; else ++g;
            } else {
                if (g == 0) dir = 1; else --g;
            }
        } else {
            g = (g + 1 == n) ? 0 : g + 1;
        }
    }
};

// The rows one stage keeps between beats, and the neighbour sums they give.
// cen = row q of the stage's input, C = row q + 1, just arrived.
//
// FP32 torus, linear sums: the cell sum is (n + w) + (s + e), and s + e of cell
// (q, j) is n + w of cell (q + 1, j + 1).  So a stage keeps row q and the
// pair sums acc(j) = row_{q-1}(j+1) + row_q(j) instead of rows q - 1 and q:
// the sum of a cell is its own new pair (row_q(j+1) + C(j)) plus the old pair
// one column to the west -- two additions per field instead of three, at the
// same registers and the same two shuffles.  4096^2, K = 8:
// 92.7 -> 82.7 us a launch.
// Zero flux and FP64: rows q - 1 and q, three additions (nbr_sum says why).
// CeNN cell (OUT): the sums run over the outputs y = clamp(x), clamped once
// when a row arrives and kept (pair sums and y of row q on the FP32 torus, y of
// rows q - 1 and q otherwise) instead of once per neighbour; v is
// constant, so it needs no sums.  4096^2, K = 8: torus 73.5 -> 57.2 us a
// launch, zero flux 75.7 -> 69.6 us.
//
// Row sets rotate by beat phase PH = m % kPhases without register moves:
// two-phase stages hold row q in row[PH] and put C into row[PH ^ 1], the
// three-phase ones hold rows q - 1, q, q + 1 in row[PH], row[PH + 1],
// row[PH + 2].
template <typename T, int V, int K, int BC, bool OUT> struct StageRows {
    static constexpr bool kPair = PairSums<BC, T>::value && K > 1;
    static constexpr int kPhases = (!kPair && !OUT) ? 3 : 2;
    Slice<T, V> row[kPhases];
    T acc[2][V];

    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int a = 0; a < kPhases; ++a) zero_slice(row[a]);
#pragma unroll
        for (int e = 0; e < V; ++e) acc[0][e] = acc[1][e] = T(0);
    }

    template <int PH>
    __device__ __forceinline__ const Slice<T, V> &cen() const {
        return kPhases == 3 ? row[(PH + 1) % 3] : row[PH];
    }
    template <int PH>
    __device__ __forceinline__ void put(const Slice<T, V> &C) {
        row[kPhases == 3 ? (PH + 2) % 3 : (PH ^ 1)] = C;
    }

    // Take in a row without computing one (light-cone fill): the stage's
    // first row, or (FIRST = false) its second.
    template <int PH, bool FIRST>
    __device__ __forceinline__ void keep(const Slice<T, V> &C) {
        if constexpr (kPhases == 2) {
            const Slice<T, V> &B = row[PH];
            if constexpr (!OUT) {
                if constexpr (!FIRST) {  // (linear two-phase stages keep pairs)
                    const T eu = __shfl_down_sync(kFull, B.u[0], 1);
                    const T ev = __shfl_down_sync(kFull, B.v[0], 1);
#pragma unroll
                    for (int e = 0; e < V; ++e) {
                        acc[0][e] = add_rn(e == V - 1 ? eu : B.u[e + 1], C.u[e]);
                        acc[1][e] = add_rn(e == V - 1 ? ev : B.v[e + 1], C.v[e]);
                    }
                }
            } else if constexpr (kPair) {
                T y[V];
#pragma unroll
                for (int e = 0; e < V; ++e) y[e] = clamp1(C.u[e]);
                if constexpr (!FIRST) {
                    const T ey = __shfl_down_sync(kFull, acc[1][0], 1);
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[0][e] = add_rn(e == V - 1 ? ey : acc[1][e + 1], y[e]);
                }
#pragma unroll
                for (int e = 0; e < V; ++e) acc[1][e] = y[e];
            } else {  // outputs of rows q - 1, q in acc[PH], acc[PH ^ 1]
#pragma unroll
                for (int e = 0; e < V; ++e) acc[PH][e] = clamp1(C.u[e]);
            }
        }
        put<PH>(C);
    }

    // The neighbour sums su, sv (and the outputs yc, OUT only) of row q; then
    // C takes its place among the kept rows (the caller calls put<PH>(C)).
    template <int PH>
    __device__ __forceinline__ void sums(const Slice<T, V> &C, T (&su)[V], T (&sv)[V], T (&yc)[V]) {
        const Slice<T, V> &B = cen<PH>();
        if constexpr (OUT) {
            T y[V];
#pragma unroll
            for (int e = 0; e < V; ++e) y[e] = clamp1(C.u[e]);
            if constexpr (kPair) {
                const T wy = __shfl_up_sync(kFull, acc[0][V - 1], 1);
                const T ey = __shfl_down_sync(kFull, acc[1][0], 1);
#pragma unroll
                for (int e = V - 1; e >= 0; --e) {
                    const T a = add_rn(e == V - 1 ? ey : acc[1][e + 1], y[e]);
                    su[e] = add_rn(e == 0 ? wy : acc[0][e - 1], a);
                    acc[0][e] = a;
                }
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    yc[e] = acc[1][e];
                    acc[1][e] = y[e];
                }
            } else {
                const T wy = __shfl_up_sync(kFull, acc[PH ^ 1][V - 1], 1);
                const T ey = __shfl_down_sync(kFull, acc[PH ^ 1][0], 1);
#pragma unroll
                for (int e = 0; e < V; ++e) {
                    su[e] = nbr_sum<BC>(acc[PH][e], y[e], e == 0 ? wy : acc[PH ^ 1][e - 1],
                                        e == V - 1 ? ey : acc[PH ^ 1][e + 1]);
                    yc[e] = acc[PH ^ 1][e];
                }
#pragma unroll
                for (int e = 0; e < V; ++e) acc[PH][e] = y[e];
            }
        } else if constexpr (kPair) {
            const T wu = __shfl_up_sync(kFull, acc[0][V - 1], 1);
            const T eu = __shfl_down_sync(kFull, B.u[0], 1);
            const T wv = __shfl_up_sync(kFull, acc[1][V - 1], 1);
            const T ev = __shfl_down_sync(kFull, B.v[0], 1);
#pragma unroll
            for (int e = V - 1; e >= 0; --e) {
                const T a = add_rn(e == V - 1 ? eu : B.u[e + 1], C.u[e]);
                const T b = add_rn(e == V - 1 ? ev : B.v[e + 1], C.v[e]);
                su[e] = add_rn(e == 0 ? wu : acc[0][e - 1], a);
                sv[e] = add_rn(e == 0 ? wv : acc[1][e - 1], b);
                acc[0][e] = a;
                acc[1][e] = b;
            }
        } else {
            const Slice<T, V> &A = row[PH];
            const T wu = __shfl_up_sync(kFull, B.u[V - 1], 1);
            const T eu = __shfl_down_sync(kFull, B.u[0], 1);
            const T wv = __shfl_up_sync(kFull, B.v[V - 1], 1);
            const T ev = __shfl_down_sync(kFull, B.v[0], 1);
#pragma unroll
            for (int e = 0; e < V; ++e) {
                su[e] = nbr_sum<BC>(A.u[e], C.u[e], e == 0 ? wu : B.u[e - 1], e == V - 1 ? eu : B.u[e + 1]);
                sv[e] = nbr_sum<BC>(A.v[e], C.v[e], e == 0 ? wv : B.v[e - 1], e == V - 1 ? ev : B.v[e + 1]);
            }
        }
    }
};

// Ring rows of a pipeline with the given number of phases.
template <int PHASES> struct RingRows : IntC<PHASES == 3 ? kRing : kRing2> {};

// One pipeline beat: take input row m of the strip from ring slot rd (issuing
// the copy of row m + R - 1 into slot wr first, R the ring's rows), advance
// every stage by one row, and hand the finished row (stage K) to the policy.
//
// The policy P supplies the per-stage arithmetic and the stores:
//   P::kOutputSum                        neighbour sums over clamp(x) (CeNN)
//   P::issue(j, slot)                    extra cp.async copies for beat j,
//                                        committed with input row j
//   P::stage(s, cen, su, sv, yc, q, slot, out)
//        stage s maps row q (cen) of its input and its neighbour sums to row
//        q of its output (q = input-row index within the strip, see
//        temporal_strip); slot = the beat's ring slot
//   P::finish(q, out)                    the row q leaving the last stage
//   P::finish_main(q, out)               the same for a beat of the main loop,
//                                        where q >= K holds: the owned row
//                                        check may be dropped
//
// CHECK = false: a beat of the main loop's whole groups of kPhases beats,
// which needs neither the end-of-strip test nor the last-copy test (measured
// at K = 8, 4096^2: 1427 -> 1448 Gcell-updates/s); the copies past the strip's
// last row are of wrapped rows of the grid and are not read.
//
// ACTIVE < K (the first 2K beats of a strip): only stages s < ACTIVE compute;
// stage ACTIVE just keeps its input row for the next beats.  Row q of the
// last stage needs stage s's rows from q - (K - 1 - s) on, and the stored
// rows have q >= K, so stage s's rows 0 .. s feed nothing that is stored.
// Beat m computes stage s's row m - s - 1, so stage s first matters at beat
// 2s + 2: ACTIVE = m / 2, and stage ACTIVE keeps its first row at beat 2s and
// its second at beat 2s + 1.
template <typename T, int K, int PH, int BC, int ACTIVE = K, bool CHECK = true, bool FIRST = false, class S, class P>
__device__ __forceinline__ void pipeline_beat(int m, int total, S (&st)[K], const RowRing<T> &ring, int rd, int wr,
                                              RowWalk<BC> &walk, int nn, int nm, const StripGeom &geo,
                                              const T *__restrict__ u, const T *__restrict__ v, P &pol) {
    constexpr int V = Vec<T>::N;
    constexpr int R = RingRows<S::kPhases>::value;
    if (CHECK && m >= total) return;
    // The slot written here was read in the previous beat, whose stage
    // computations (issued before this point) consumed that value.
    if (!CHECK || m + R - 1 < total) {
        ring_issue_at(ring, wr, walk.g, nm, geo, u, v);
        walk.next(nn);
        pol.issue(m + R - 1, wr);
    }
    cp_async_commit();
    cp_async_wait<R - 1>();  // the group holding row m is complete
    Slice<CT<T>, V> cur;
    ring_read_bc<T, BC>(ring, rd, geo.rev, cur);
#pragma unroll
    for (int s = 0; s < K; ++s) {
        if (s < ACTIVE) {
            CT<T> su[V], sv[V], yc[V];
            st[s].template sums<PH>(cur, su, sv, yc);
            Slice<CT<T>, V> out;
            pol.stage(s, st[s].template cen<PH>(), su, sv, yc, m - s - 1, rd, out);
            st[s].template put<PH>(cur);
            cur = out;
        } else if (s == ACTIVE) {
            st[s].template keep<PH, FIRST>(cur);  // stage s - 1's row, needed from the next beat on
        }
    }
    if constexpr (ACTIVE == K) {
        if constexpr (CHECK) pol.finish(m - K, cur);
        else pol.finish_main(m - K, cur);
    }
}

// The first 2K beats of a strip (ACTIVE = M / 2), unrolled at compile time.
template <typename T, int K, int BC, int M, class S, class P>
__device__ __forceinline__ void pipeline_fill(int total, S (&st)[K], const RowRing<T> &ring, RowWalk<BC> &walk,
                                              int nn, int nm, const StripGeom &geo, const T *__restrict__ u,
                                              const T *__restrict__ v, P &pol) {
    constexpr int R = RingRows<S::kPhases>::value;
    pipeline_beat<T, K, M % S::kPhases, BC, (M / 2 < K ? M / 2 : K), true, M % 2 == 0>(
        M, total, st, ring, M % R, (M + R - 1) % R, walk, nn, nm, geo, u, v, pol);
    if constexpr (M + 1 < 2 * K)
        pipeline_fill<T, K, BC, M + 1>(total, st, ring, walk, nn, nm, geo, u, v, pol);
}

template <typename T, int K, int H, int BC = BC_WRAP>
__device__ __forceinline__ StripGeom strip_geom(int band, int strip, int nn, int nm, int rows) {
    constexpr int V = Vec<T>::N;
    static_assert(H * V >= K, "halo narrower than the temporal depth");
    static_assert(2 * H < 32, "halo wider than the warp");
    constexpr int OUTW = (32 - 2 * H) * V;
    const int lane = threadIdx.x & 31;
    StripGeom g;
    const int c0 = band * OUTW;
    const int64_t c = (int64_t)c0 - H * V + lane * V;
    g.rev = false;
    if constexpr (IsRagged<T>::value) {
#pragma unroll
        for (int e = 0; e < V; ++e) g.col[e] = bc_index<BC>((int64_t)c0 - H * V + lane + 32 * e, nm);
    } else if constexpr (BC == BC_MIRROR) {
        // columns c .. c+V-1 of the 2NM-periodic mirror image: inside the
        // grid, or the reversed vector starting at 2NM - V - q (V-aligned)
        const int q = wrap_row(c, 2 * (int64_t)nm);
        g.rev = q >= nm;
        g.lc = g.rev ? 2 * nm - V - q : q;
    } else {
        g.lc = wrap_row(c, nm);  // V-aligned since nm % V == 0
    }
    g.sc = c0 + (lane - H) * V;
    g.st_lane = (lane >= H) && (lane < 32 - H) && (g.sc < nm);
    g.nel = min(V, nm - g.sc);
    g.r0 = strip * rows;
    g.nout = min(rows, nn - g.r0);
    g.total = g.nout + 2 * K;
    return g;
}

// Run one work item through the K-stage pipeline: input rows of (u, v) pass
// through the stages; the policy decides what each stage computes and stores.
// Every policy stores (or sums over) owned rows only, q >= K, so the first 2K
// beats skip the stages outside their light cone.
template <typename T, int K, int BC = BC_WRAP, class P>
__device__ __forceinline__ void pipeline_strip(const StripGeom &geo, const T *__restrict__ u,
                                               const T *__restrict__ v, int nn, int nm, P &pol) {
    typedef StageRows<CT<T>, Vec<T>::N, K, BC, P::kOutputSum> S;
    constexpr int N = S::kPhases;
    constexpr int R = RingRows<N>::value;
    S st[K];
#pragma unroll
    for (int s = 0; s < K; ++s) st[s].zero();

    typedef typename Vec<T>::type VT;
    __shared__ __align__(16) VT ring_mem[kTemporalWarps][R][2][32];
    RowRing<T> ring;
    ring.slot = ring_mem[(threadIdx.x >> 5) % kTemporalWarps];

    // prologue: rows 0 .. R-2 in flight, one commit group each
    RowWalk<BC> walk;
    walk.start((int64_t)geo.r0 - K, nn);
#pragma unroll
    for (int j = 0; j < R - 1; ++j) {
        if (j < geo.total) {
            ring_issue_at(ring, j, walk.g, nm, geo, u, v);
            walk.next(nn);
            pol.issue(j, j);
        }
        cp_async_commit();
    }
    // a strip has total = nout + 2K > 2K beats, so the fill always completes
    constexpr int M0 = 2 * K;
    pipeline_fill<T, K, BC, 0>(geo.total, st, ring, walk, nn, nm, geo, u, v, pol);
    int m = M0;
    if constexpr (N == 3) {
        for (; m + 2 < geo.total; m += 3) {  // whole triplets: no per-beat bounds tests
            pipeline_beat<T, K, M0 % 3, BC, K, false>(m, geo.total, st, ring, M0 % 3, (M0 + 2) % 3, walk, nn, nm,
                                                      geo, u, v, pol);
            pipeline_beat<T, K, (M0 + 1) % 3, BC, K, false>(m + 1, geo.total, st, ring, (M0 + 1) % 3, M0 % 3, walk,
                                                            nn, nm, geo, u, v, pol);
            pipeline_beat<T, K, (M0 + 2) % 3, BC, K, false>(m + 2, geo.total, st, ring, (M0 + 2) % 3, (M0 + 1) % 3,
                                                            walk, nn, nm, geo, u, v, pol);
        }
        // the last 0 .. 2 beats
        pipeline_beat<T, K, M0 % 3, BC>(m, geo.total, st, ring, M0 % 3, (M0 + 2) % 3, walk, nn, nm, geo, u,
                                        v, pol);
        pipeline_beat<T, K, (M0 + 1) % 3, BC>(m + 1, geo.total, st, ring, (M0 + 1) % 3, M0 % 3, walk, nn, nm, geo, u, v, pol);
    } else {
        int rd = M0 % R;  // even; row m sits in slot m % R
        for (; m + 1 < geo.total; m += 2) {  // whole pairs: no per-beat bounds tests
            pipeline_beat<T, K, 0, BC, K, false>(m, geo.total, st, ring, rd, (rd + R - 1) % R, walk, nn, nm, geo, u, v, pol);
            pipeline_beat<T, K, 1, BC, K, false>(m + 1, geo.total, st, ring, rd + 1, rd, walk, nn, nm, geo,
                                                 u, v, pol);
            rd = (rd + 2) % R;
        }
        // the last 0 or 1 beats
        pipeline_beat<T, K, 0, BC>(m, geo.total, st, ring, rd, (rd + R - 1) % R, walk, nn, nm, geo, u, v,
                                   pol);
    }
    cp_async_wait<0>();
}

// Forward policy: Eq. 1 at every stage; the last stage's owned rows are stored.
template <typename T, int K, int RX>
struct ForwardPolicy {
    static constexpr bool kOutputSum = (RX == RX_CENN);
    const Coef<CT<T>> &p;
    const StripGeom &geo;
    T *__restrict__ un;
    T *__restrict__ vn;
    int nm;
    __device__ __forceinline__ void issue(int, int) {}
    __device__ __forceinline__ void stage(int, const Slice<CT<T>, Vec<T>::N> &cen, const CT<T> (&su)[Vec<T>::N],
                                          const CT<T> (&sv)[Vec<T>::N], const CT<T> (&yc)[Vec<T>::N], int, int,
                                          Slice<CT<T>, Vec<T>::N> &out) {
        slice_react<CT<T>, RX, Vec<T>::N>(cen, su, sv, yc, p, out);
    }
    __device__ __forceinline__ void finish(int q, const Slice<CT<T>, Vec<T>::N> &out) {
        const int orow = q - K;
        if (orow >= 0) {  // the same for the whole warp
            const int64_t off = (int64_t)(geo.r0 + orow) * nm + geo.sc;
            store(off, out);
        }
    }
    __device__ __forceinline__ void finish_main(int q, const Slice<CT<T>, Vec<T>::N> &out) {
        store((int64_t)(geo.r0 + q - K) * nm + geo.sc, out);
    }
    __device__ __forceinline__ void store(int64_t off, const Slice<CT<T>, Vec<T>::N> &out) {
        if (!geo.st_lane) return;
        if constexpr (IsRagged<T>::value) {
#pragma unroll
            for (int e = 0; e < Vec<T>::N; ++e) {
                if (e < geo.nel) {
                    un[off + e].x = out.u[e];
                    vn[off + e].x = out.v[e];
                }
            }
        } else {
            store_vec<T>(un + off, out.u);
            store_vec<T>(vn + off, out.v);
        }
    }
};

// Planes of the K intermediate states written by ForwardAllPolicy.
template <typename T> struct StagePlanes {
    T *u[8];
    T *v[8];
};

// Forward policy that also stores the owned rows of every stage s (the state
// s+1 steps ahead) into planes.u[s], planes.v[s]: the states a reverse sweep
// needs, K per launch.
template <typename T, int K, int RX>
struct ForwardAllPolicy {
    static constexpr bool kOutputSum = (RX == RX_CENN);
    const Coef<CT<T>> &p;
    const StripGeom &geo;
    const StagePlanes<T> &planes;
    int nm;
    __device__ __forceinline__ void issue(int, int) {}
    __device__ __forceinline__ void stage(int s, const Slice<CT<T>, Vec<T>::N> &cen, const CT<T> (&su)[Vec<T>::N],
                                          const CT<T> (&sv)[Vec<T>::N], const CT<T> (&yc)[Vec<T>::N], int q, int,
                                          Slice<CT<T>, Vec<T>::N> &out) {
        slice_react<CT<T>, RX, Vec<T>::N>(cen, su, sv, yc, p, out);
        const int orow = q - K;
        if (orow >= 0 && orow < geo.nout && geo.st_lane) {
            const int64_t off = (int64_t)(geo.r0 + orow) * nm + geo.sc;
            store_vec<T>(planes.u[s] + off, out.u);
            store_vec<T>(planes.v[s] + off, out.v);
        }
    }
    __device__ __forceinline__ void finish(int, const Slice<CT<T>, Vec<T>::N> &) {}
    __device__ __forceinline__ void finish_main(int, const Slice<CT<T>, Vec<T>::N> &) {}
};

// H = halo lanes per side; any H >= ceil(K/V) is correct (a larger H than
// needed only narrows the band), which lets a batched launch use one band
// layout for launches of different depth.
template <typename T, int K, int H, int RX, int BC = BC_WRAP>
__device__ __forceinline__ void temporal_strip(int band, int strip, const T *__restrict__ u,
                                               const T *__restrict__ v, T *__restrict__ un,
                                               T *__restrict__ vn, int nn, int nm, int rows,
                                               const Coef<CT<T>> &p) {
    const StripGeom geo = strip_geom<T, K, H, BC>(band, strip, nn, nm, rows);
    ForwardPolicy<T, K, RX> pol{p, geo, un, vn, nm};
    pipeline_strip<T, K, BC>(geo, u, v, nn, nm, pol);
}

constexpr int kTemporalBlock = 32 * kTemporalWarps;

// The single-grid temporally blocked kernel: warp w of the launch owns work
// item (band w % bands, strip w / bands).
template <typename T, int K, int RX, int BC>
__global__ void __launch_bounds__(kTemporalBlock)
k_temporal(const T *__restrict__ u, const T *__restrict__ v, T *__restrict__ un,
           T *__restrict__ vn, int nn, int nm, int bands, int nwarps, int rows, Coef<CT<T>> p) {
    pdl_wait();
    const int wid = blockIdx.x * (kTemporalBlock / 32) + (threadIdx.x >> 5);
    if (wid >= nwarps) return;  // whole warps only
    constexpr int H = (K + Vec<T>::N - 1) / Vec<T>::N;
    temporal_strip<T, K, H, RX, BC>(wid % bands, wid / bands, u, v, un, vn, nn, nm, rows, p);
    pdl_trigger();
}

}  // namespace rdk
