// forward.cu -- forward kernels for Eq. 1-3 (Sec. II.A) and the launchers of
// every forward variant (torus or zero flux; FitzHugh-Nagumo, pure diffusion
// or CeNN cell; float / double planes, or bf16 / half planes computed in FP32).
//
//  k_step1     one time step per launch (float / double planes).  A warp owns a band of 32*V columns
//              (V = 4 floats / 2 doubles per lane, one 16-byte load) and walks
//              down a strip of rows, keeping rows i-1, i, i+1 in registers and
//              prefetching row i+2.  Horizontal neighbours come from the
//              adjacent lane by warp shuffle; the two band-edge values are
//              read from global memory (L1/L2 hits).  Each input byte is read
//              once from DRAM and each output byte written once: 16 B per
//              cell-step in FP32, the algorithmic minimum.
//  k_temporal  K time steps per launch.  A warp loads a band of 32*V columns
//              that overlaps its neighbours by H = ceil(K/V) lanes on each
//              side, and walks down rows r0-K .. r0+R+K-1 of its strip.  Stage
//              s of a K-deep register pipeline turns three rows of stage s-1
//              into one row of stage s, so a row is read once and leaves as
//              K-step-advanced output: DRAM traffic is 16 B per cell per K
//              steps.  Lanes within K columns of the band edge hold stale
//              values after K steps and do not store.
//  k_generic   one thread per cell, scalar loads: any size and alignment.
//              (AUTO takes it for 16-bit and FP64 planes only; FP32 planes that
//              are not vector-aligned run k_temporal on Ragged rows.)
//
// All three evaluate cells with rdk::nbr_sum and rdk::cell_react, so they produce identical
// bits for identical inputs (for 16-bit planes: at the same steps per
// launch, which is also the rounding interval).  Under the zero-flux boundary the single-step
// and generic kernels clamp neighbour indices into the grid (the ghost cell
// is the edge cell); the temporal kernel loads mirrored halos instead
// (temporal.cuh).  k_temporal's launchers live in temporal_launch.cuh and are
// instantiated in the temporal_*.cu units, the warp-pair variant's
// (k_temporal_split) in split_launch.cuh and the split_*.cu units; they
// compile in parallel.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "internal.h"
#include "temporal.cuh"
#include "split_launch.cuh"

// the warp-pair kernels compile in split_f32a.cu .. split_f32c.cu and split_f64.cu
RDK_EXTERN_SPLIT(float, 2) RDK_EXTERN_SPLIT(float, 3) RDK_EXTERN_SPLIT(float, 4) RDK_EXTERN_SPLIT(float, 5)
RDK_EXTERN_SPLIT(float, 6) RDK_EXTERN_SPLIT(float, 7) RDK_EXTERN_SPLIT(float, 8)
RDK_EXTERN_SPLIT(double, 2) RDK_EXTERN_SPLIT(double, 3) RDK_EXTERN_SPLIT(double, 4)

namespace rdk {

namespace {

// 72 registers.  4096^2 FP32, 400 back-to-back launches (Gcell-updates/s; 2 / 4 / 8 rows per warp):
// 32 threads 245 / 389 / 372, 64 threads 398 / 392 / 364, 128 threads 393 / 393 / 362,
// 256 threads 369 / 385 / 345.
constexpr int kStep1Block = 64;

// --------------------------------------------------------------------------- single step

// FP32 / FP64 planes (16-bit planes take the ring-staged pipeline at k = 1,
// see step1_t).
template <typename T, int RX, int BC>
__global__ void __launch_bounds__(kStep1Block)
k_step1(const T *__restrict__ u, const T *__restrict__ v, T *__restrict__ un,
        T *__restrict__ vn, int nn, int nm, int bands, int nwarps, int rows, Coef<T> p) {
    constexpr int V = Vec<T>::N;
    constexpr bool zf = (BC == BC_MIRROR);
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int wid = blockIdx.x * (kStep1Block / 32) + (threadIdx.x >> 5);
    if (wid >= nwarps) return;  // whole warps only
    const int band = wid % bands;
    const int strip = wid / bands;
    const int col = band * 32 * V + lane * V;
    const bool active = col < nm;
    // neighbour columns beyond the edges: wrapped, or the edge cell itself
    const int colw = (col == 0) ? (zf ? 0 : nm - 1) : col - 1;
    const int cole = (col + V >= nm) ? (zf ? nm - 1 : 0) : col + V;
    const bool edge_w = (lane == 0);
    const bool edge_e = active && (lane == 31 || col + V >= nm);
    const int r0 = strip * rows;
    const int r1 = min(r0 + rows, nn);

    Slice<T> nor, cen, sou, pre;
    T cw_u = 0, ce_u = 0, cw_v = 0, ce_v = 0;  // band-edge values of row "cen"
    T sw_u = 0, se_u = 0, sw_v = 0, se_v = 0;  // ... of row "sou"
    T pw_u = 0, pe_u = 0, pw_v = 0, pe_v = 0;  // ... of row "pre"
    zero_slice(nor); zero_slice(cen); zero_slice(sou); zero_slice(pre);

    int rn = (r0 == 0) ? (zf ? 0 : nn - 1) : r0 - 1;
    int rc = r0;
    int rs = (r0 + 1 == nn) ? (zf ? nn - 1 : 0) : r0 + 1;
    if (active) {
        load_slice(nor, u, v, (int64_t)rn * nm + col);
        load_slice(cen, u, v, (int64_t)rc * nm + col);
        load_slice(sou, u, v, (int64_t)rs * nm + col);
    }
    if (edge_w) {
        cw_u = __ldg(u + (int64_t)rc * nm + colw); cw_v = __ldg(v + (int64_t)rc * nm + colw);
        sw_u = __ldg(u + (int64_t)rs * nm + colw); sw_v = __ldg(v + (int64_t)rs * nm + colw);
    }
    if (edge_e) {
        ce_u = __ldg(u + (int64_t)rc * nm + cole); ce_v = __ldg(v + (int64_t)rc * nm + cole);
        se_u = __ldg(u + (int64_t)rs * nm + cole); se_v = __ldg(v + (int64_t)rs * nm + cole);
    }

    for (int r = r0; r < r1; ++r) {
        // prefetch row r+2 (wrapped) while row r is computed
        const bool more = (r + 1 < r1);
        const int rp = (rs + 1 == nn) ? (zf ? nn - 1 : 0) : rs + 1;
        if (more) {
            if (active) load_slice(pre, u, v, (int64_t)rp * nm + col);
            if (edge_w) { pw_u = __ldg(u + (int64_t)rp * nm + colw); pw_v = __ldg(v + (int64_t)rp * nm + colw); }
            if (edge_e) { pe_u = __ldg(u + (int64_t)rp * nm + cole); pe_v = __ldg(v + (int64_t)rp * nm + cole); }
        }
        T wu = __shfl_up_sync(kFull, cen.u[V - 1], 1);
        T eu = __shfl_down_sync(kFull, cen.u[0], 1);
        T wv = __shfl_up_sync(kFull, cen.v[V - 1], 1);
        T ev = __shfl_down_sync(kFull, cen.v[0], 1);
        if (edge_w) { wu = cw_u; wv = cw_v; }
        if (edge_e) { eu = ce_u; ev = ce_v; }
        Slice<T> out;
        slice_update<T, RX, BC>(nor, cen, sou, wu, eu, wv, ev, p, out);
        if (active) {
            const int64_t off = (int64_t)r * nm + col;
            store_vec<T>(un + off, out.u);
            store_vec<T>(vn + off, out.v);
        }
        nor = cen; cen = sou; sou = pre;
        cw_u = sw_u; ce_u = se_u; cw_v = sw_v; ce_v = se_v;
        sw_u = pw_u; se_u = pe_u; sw_v = pw_v; se_v = pe_v;
        rs = rp;
    }
    pdl_trigger();
}

// --------------------------------------------------------------------------- temporal blocking

// --------------------------------------------------------------------------- generic

template <typename T, int RX, int BC>
__global__ void __launch_bounds__(256)
k_generic(const T *__restrict__ u, const T *__restrict__ v, T *__restrict__ un,
          T *__restrict__ vn, int nn, int nm, Coef<CT<T>> p) {
    constexpr bool zf = (BC == BC_MIRROR);
    pdl_wait();
    const int64_t n = (int64_t)nn * nm;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(idx / nm);
        const int j = (int)(idx - (int64_t)i * nm);
        const int ip = (i + 1 == nn) ? (zf ? i : 0) : i + 1;
        const int im = (i == 0) ? (zf ? 0 : nn - 1) : i - 1;
        const int jp = (j + 1 == nm) ? (zf ? j : 0) : j + 1;
        const int jm = (j == 0) ? (zf ? 0 : nm - 1) : j - 1;
        const int64_t ri = (int64_t)i * nm;
        const int64_t rp = (int64_t)ip * nm;
        const int64_t rm = (int64_t)im * nm;
        CT<T> ou, ov;
        cell_update<CT<T>, RX, BC>(load1(u + ri + j), load1(u + rm + j), load1(u + rp + j), load1(u + ri + jm),
                               load1(u + ri + jp), load1(v + ri + j), load1(v + rm + j), load1(v + rp + j),
                               load1(v + ri + jm), load1(v + ri + jp), p, ou, ov);
        un[idx] = to_storage<T>(ou);
        vn[idx] = to_storage<T>(ov);
    }
    pdl_trigger();
}

template <typename T>
__global__ void __launch_bounds__(256)
k_init(const T *x, T *u, T *v, CT<T> ka, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const T t = to_storage<T>(mul_rn(ka, to_compute<T>(x[i])));  // x may alias u: plain loads
        u[i] = t;
        v[i] = t;
    }
}

// du = su, dv = sv, n vectors of 16 bytes each; one read where su == sv.
__global__ void __launch_bounds__(256)
k_copy_planes(const uint4 *__restrict__ su, const uint4 *__restrict__ sv, uint4 *__restrict__ du, uint4 *__restrict__ dv,
              int64_t n) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint4 x = __ldg(su + i);
        const uint4 y = su == sv ? x : __ldg(sv + i);
        du[i] = x;
        dv[i] = y;
    }
    pdl_trigger();
}

template <typename T>
cudaError_t step1_t(int reaction, int boundary, const void *u, const void *v, void *un, void *vn,
                    int64_t nn, int64_t nm, const rdcnn_params &p, int rows, cudaStream_t s) {
    if constexpr (!is_f32_f64<T>()) {
        // 16-bit planes: a row carries half the bytes, and keeping HBM busy needs
        // more rows in flight than the register prefetch above holds; the
        // cp.async ring of the temporal pipeline at depth 1 keeps three per warp
        // (same arithmetic, one rounding per step: the same bits), with 8 values
        // (16 bytes) per lane when NM and the alignment allow.
        if (nm % 8 == 0 && aligned16(u) && aligned16(v) && aligned16(un) && aligned16(vn))
            return temporal_launch<Wide<T>, 1>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
        return temporal_launch<T, 1>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
    } else {
        constexpr int V = Vec<T>::N;
        const int bands = (int)((nm + 32 * V - 1) / (32 * V));
        const int strips = (int)((nn + rows - 1) / rows);
        const int64_t nwarps = (int64_t)bands * strips;
        const int wpb = kStep1Block / 32;
        const unsigned grid = (unsigned)((nwarps + wpb - 1) / wpb);
        const Coef<T> c = make_coef<T>(p, reaction);
        return with_model(reaction, boundary, [&](auto rx, auto bc) {
            const cudaError_t e = launch_k(k_step1<T, decltype(rx)::value, decltype(bc)::value>, grid,
                                           kStep1Block, 0, s, (const T *)u, (const T *)v, (T *)un, (T *)vn,
                                           (int)nn, (int)nm, bands, (int)nwarps, rows, c);
            count_launches(1);
            return e;
        });
    }
}

}  // namespace

// Launch shape of the FP32 temporal pipeline, rows per warp and depth, from a
// model of a launch: a warp's strip of R rows is R beats and a fill of f k more,
// and a beat takes a + b k us with one warp on each of an SM's four schedulers,
// a2 + b2 k with two (which is what the registers of k = 8 allow); more warps
// run in waves of that.  So only a few strip lengths can be best for a depth:
// those with which the warps just fill one warp per scheduler, two, or w waves.
// Fitted (us) to a sweep of k = 3 .. 8 and 25 strip lengths at 18 shapes from
// 300^2 to 4096^2, FitzHugh-Nagumo on the torus and under zero flux, CeNN under
// zero flux: the shape it picks is within 1.1 % of the best one measured (7 % at
// most), the size classes before it (k = 4, 6, 8; 4 or 16 rows below 2^22 cells)
// were 17 % off on average and up to 68 %.  us a step, before / now: 384^2
// 1.18 / 0.95, 768^2 1.51 / 1.30, 1536^2 3.47 / 2.45, 3072^2 8.03 / 6.33, 4096 x
// 1024 4.56 / 3.62, 1024^2 and 4096^2 unchanged.  Ragged rows cost more per beat
// (single elements are copied), so their depths begin at 5: 14 shapes, 3.2 % off
// the best on average (13 % at most), before 22 %.
namespace {

struct BeatModel {
    double launch, a, b, f, a2, b2, f2;
    int k0, k1;  // depths AUTO chooses among
};
constexpr BeatModel kBeats = {1.680, 0.0764, 0.0394, 2.690, 0.0692, 0.0548, 1.823, 4, 8};
constexpr BeatModel kRaggedBeats = {1.692, 0.2179, 0.0290, 3.830, 0.1335, 0.0829, 1.714, 5, 8};

// us of a launch of depth K with `warps` strips of `rows` rows.
double launch_us(const BeatModel &m, int K, int64_t warps, int64_t rows, int64_t slots) {
    if (warps <= slots / 2) return m.launch + (m.a + m.b * K) * ((double)rows + m.f * K);
    return m.launch + (double)((warps + slots - 1) / slots) * (m.a2 + m.b2 * K) * ((double)rows + m.f2 * K);
}

// Best rows for depth K; *us: what a launch then takes.
int model_rows(const BeatModel &m, int K, int64_t nn, int64_t nm, double *us) {
    const int H = (K + 3) / 4;
    const int64_t bands = (nm + (32 - 2 * H) * 4 - 1) / ((32 - 2 * H) * 4);
    const int64_t slots = (int64_t)sm_count() * 8;
    int best = 1;
    int64_t strips = 0;
    *us = 1e300;
    for (int w = 0; w <= 8 && strips < (nn + 1) / 2; ++w) {  // w = 0: one warp per scheduler
        strips = std::min<int64_t>((w ? w * slots : slots / 2) / bands, (nn + 1) / 2);
        if (strips < 1) continue;
        const int64_t rows = (nn + strips - 1) / strips;
        const double t = launch_us(m, K, bands * ((nn + rows - 1) / rows), rows, slots);
        if (t < *us) { *us = t; best = (int)rows; }
    }
    if (*us > 1e299) best = 256;  // more bands than the waves looked at hold
    return best;
}

int model_depth(const BeatModel &m, int64_t nn, int64_t nm) {
    int best = m.k1;
    double least = 1e300;
    for (int K = m.k0; K <= m.k1; ++K) {
        double us;
        (void)model_rows(m, K, nn, nm, &us);
        if (us / K < least) { least = us / K; best = K; }
    }
    return best;
}

}  // namespace

double temporal_us(int K, int64_t warps, int64_t rows, int sms) { return launch_us(kBeats, K, warps, rows, (int64_t)sms * 8); }

int auto_rows_f32(bool ragged, int K, int64_t nn, int64_t nm) {
    double us;
    return model_rows(ragged ? kRaggedBeats : kBeats, K, nn, nm, &us);
}

// Depths up to 4 of grids whose four planes do not fit L2 together are bound by
// DRAM, not by the beats of the model: fastest with short strips at depths 1 and
// 2, and with one wave of 12 warps an SM at 3 and 4 (at 4, 16 where registers allow
// that many).  us a step, strips before the model / by the model / now: 8192^2 depth 1
// 194 / 184 / 169, 3 59 / 65 / 59, 4 48 / 60 / 44, zero flux 48 / 45 / 45; 6000^2 1 101 /
// 107 / 93, 4 24.9 / 26.1 / 24.8, zero flux 24.9 / 28.9 / 24.7; 4096^2 1 49 / 52 / 46, 4
// 13.2 / 12.9 / 11.8; 2900 x 3128 1 25.6 / 29.0 / 24.7.
bool beyond_l2(int64_t nn, int64_t nm) { return nn * nm >= 6000000; }
int dram_rows_f32(int K, int64_t nn, int64_t nm, int warps_per_sm) {
    if (K == 1) return 10;
    if (K == 2) return 12;
    if (K == 3 && nn * nm >= (int64_t(1) << 27)) return 20;
    const int64_t strips = (int64_t)warps_per_sm * sm_count() / ((nm + 119) / 120);
    return (int)(strips < 1 ? std::min<int64_t>(nn, 128) : (nn + strips - 1) / strips);
}

// us of an FP32 temporal launch at the strips it gets, and of a copy of the state.
namespace {
double launch_cost(bool ragged, int K, int64_t nn, int64_t nm) {
    const double pass = (double)(nn * nm) * 16;  // bytes of one over the planes
    if (beyond_l2(nn, nm) && K <= 4) return pass / (K == 1 ? 6.4e6 : 6.0e6);
    double us;
    (void)model_rows(ragged ? kRaggedBeats : kBeats, K, nn, nm, &us);
    if (!beyond_l2(nn, nm)) return us;
    const double dram = pass / 6.2e6;
    return std::max(us, dram) + 0.25 * std::min(us, dram);
}
// Planes that are no whole vectors are copied one after the other.
double copy_cost(int64_t nn, int64_t nm) {
    return (nn * nm % 4 != 0 ? 10.0 : 1.7) + (double)(nn * nm) * 16 / (beyond_l2(nn, nm) ? 6.2e6 : 12e6);
}
}  // namespace

// A stretch of up to 16 steps takes as many launches as cost least, the copy of a
// state that ends in the scratch planes included; a longer one launches of the
// default depth k.  home: what the parity of the number of launches must be for
// the state to end where it belongs (0 even, 1 odd; -1: anywhere).  us, launches of
// at most depth k, even in number / as here: 512^2 9 steps 18.5 / 13.4, 1024^2 9 steps 20.0 /
// 17.6, 8192^2 3 steps 375 / 348, 200000 x 4 2 steps 91 / 57.
int64_t stretch_launches(bool ragged, int64_t nn, int64_t nm, int64_t steps, int k, int home, double *us) {
    const BeatModel &m = ragged ? kRaggedBeats : kBeats;
    int64_t n = (steps + k - 1) / k;
    auto strays = [&](int64_t c) { return home >= 0 && c % 2 != home; };
    if (steps > 2 * m.k1) {
        if (strays(n) && n < steps) ++n;
        if (us) *us = (double)n * std::max(kHostUs, launch_cost(ragged, (int)((steps + n - 1) / n), nn, nm));
        return n;
    }
    double least = 1e300;
    int64_t best = n;
    for (int64_t c = (steps + m.k1 - 1) / m.k1; c <= std::min(steps, n + (strays(n) ? 1 : 0)); ++c) {
        const int K = (int)(steps / c), deeper = (int)(steps % c);  // launches of depth K + 1, the others of K
        const double t = (double)(c - deeper) * std::max(kHostUs, launch_cost(ragged, K, nn, nm)) +
                         (deeper ? deeper * std::max(kHostUs, launch_cost(ragged, K + 1, nn, nm)) : 0.0) +
                         (strays(c) ? std::max(kHostUs, copy_cost(nn, nm)) : 0.0);
        if (t <= least) { least = t; best = c; }
    }
    if (us) *us = least;
    return best;
}

// Whether AUTO steps FP32 rows that are no lane vectors through the pipeline
// rather than one thread a cell.  The pipeline's warps are 128 columns wide
// whatever the grid's width, so narrow tall grids are better off with threads,
// the more so the fewer steps there are (a pass over memory then advances few of
// them, and one or two also need fuller bands).  us for 24 steps, threads /
// pipeline: 200000 x 1 62 / 1080, 200000 x 3 127 / 511, 100000 x 13 225 / 223, 100000 x
// 17 269 / 224, 1025 x 3 54 / 33; 3 steps: 400000 x 21 161 / 197; 2 steps: 100000 x 17 22 / 48,
// 100000 x 45 51 / 50, 20000 x 121 29 / 42, 20000 x 225 51 / 43; 1 step: 100000 x 65 50 / 57.
bool ragged_pays(int64_t nn, int64_t nm, int64_t steps) {
    if (steps > 2) return (nm - 13) * steps >= 38 || nn <= 900 * nm;
    const int64_t bands = (nm + 119) / 120;
    return nm >= (bands > 1 ? 95 * bands : steps == 2 ? 50 : 75);
}

// Rows per warp strip when the caller gives none (FP64 and 16-bit planes, 8
// values per lane, warp pairs).  Small grids use short strips (few warps exist at all); large grids pick, among a few lengths,
// the one that minimises waves x (rows + 2K) -- the work of the slowest SM
// when every resident warp slot is busy -- so a launch does not spill a
// nearly empty second wave (e.g. 4096^2, K=8: 128 rows = 1184 warps, one
// wave on 152 SMs at 8 warps each; 112 rows = 1369 warps, two waves).  The size
// classes were measured with FP32 planes, whose lanes 16-bit planes and warp pairs
// share (256^2 .. 2048^2, with the light-cone fill: 512^2, k = 6, 4 rows 150 Gcell/s, 8 rows
// 127); FP32 with 4 values per lane has had the launch model above since.
int auto_rows_temporal(int K, int64_t nn, int64_t nm, int bands, int blocks_per_sm,
                       int warps_per_block) {
    const int64_t cells = nn * nm;
    if (cells < (int64_t(1) << 19)) return 4;
    if (cells < (int64_t(1) << 22)) return 16;
    const int64_t cap = (int64_t)sm_count() * std::max(1, blocks_per_sm) * warps_per_block;
    static const int cand[] = {32, 48, 64, 96, 128, 160, 192, 256};
    int best = 64;
    double best_cost = 1e300;
    for (int r : cand) {
        const int64_t warps = (int64_t)bands * ((nn + r - 1) / r);
        const int64_t waves = (warps + cap - 1) / cap;
        const double cost = (double)waves * (double)(std::min<int64_t>(r, nn) + 2 * K);
        if (cost < best_cost) { best_cost = cost; best = r; }
    }
    return best;
}

namespace {

template <typename T>
cudaError_t generic_t(int reaction, int boundary, const void *u, const void *v, void *un, void *vn,
                      int64_t nn, int64_t nm, const rdcnn_params &p, cudaStream_t s) {
    const int64_t n = nn * nm;
    const int64_t want = (n + 255) / 256;
    const unsigned grid = (unsigned)std::min<int64_t>(want, (int64_t)sm_count() * 16);
    const Coef<CT<T>> c = make_coef<CT<T>>(p, reaction);
    return with_model(reaction, boundary, [&](auto rx, auto bc) {
        const cudaError_t e = launch_k(k_generic<T, decltype(rx)::value, decltype(bc)::value>, grid, 256, 0, s,
                                       (const T *)u, (const T *)v, (T *)un, (T *)vn, (int)nn, (int)nm, c);
        count_launches(1);
        return e;
    });
}

}  // namespace

int sm_count() {
    static std::atomic<int> known[64];  // by device
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) {
        if (dev < 64 && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) {
            if (dev < 64) known[dev].store(n, std::memory_order_relaxed);
            return n;
        }
    }
    (void)cudaGetLastError();
    return 152;
}

cudaError_t launch_step1(int dtype, int reaction, int boundary, const void *u, const void *v,
                         void *un, void *vn, int64_t nn, int64_t nm, const rdcnn_params &p, int rows,
                         cudaStream_t s) {
    return with_dtype(dtype, [&](auto tag) {
        return step1_t<decltype(tag)>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
    });
}

cudaError_t launch_temporal(int dtype, int reaction, int boundary, int k, const void *u,
                            const void *v, void *un, void *vn, int64_t nn, int64_t nm,
                            const rdcnn_params &p, int rows, cudaStream_t s) {
    return with_dtype(dtype, [&](auto tag) {
        using T = decltype(tag);
        return with_depth(k, [&](auto kk) -> cudaError_t {
            constexpr int K = decltype(kk)::value;
            if constexpr (K <= MaxDepth<T>::value)
                return temporal_launch<T, K>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
            else
                return cudaErrorInvalidValue;
        });
    });
}

cudaError_t launch_temporal_wide(int dtype, int reaction, int boundary, int k, const void *u,
                                 const void *v, void *un, void *vn, int64_t nn, int64_t nm,
                                 const rdcnn_params &p, int rows, cudaStream_t s) {
    if (dtype == RDCNN_F64) return cudaErrorInvalidValue;
    return with_dtype(dtype, [&](auto tag) {
        using T = decltype(tag);
        return with_depth(k, [&](auto kk) -> cudaError_t {
            constexpr int K = decltype(kk)::value;
            if constexpr (K <= kMaxKWide && !std::is_same<T, double>::value)
                return temporal_launch<Wide<T>, K>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
            else
                return cudaErrorInvalidValue;
        });
    });
}

// FP32 planes (the caller checks).
cudaError_t launch_temporal_ragged(int reaction, int boundary, int k, const void *u, const void *v, void *un,
                                   void *vn, int64_t nn, int64_t nm, const rdcnn_params &p, int rows,
                                   cudaStream_t s) {
    return with_depth(k, [&](auto kk) {
        return temporal_launch<Ragged<float>, decltype(kk)::value>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
    });
}

// FP32 / FP64 storage (the caller checks), every model.
cudaError_t launch_temporal_split(int dtype, int reaction, int boundary, int k, const void *u, const void *v,
                                  void *un, void *vn, int64_t nn, int64_t nm, const rdcnn_params &p,
                                  int rows, cudaStream_t s) {
    if (dtype != RDCNN_F32 && dtype != RDCNN_F64) return cudaErrorInvalidValue;
    return with_dtype(dtype, [&](auto tag) {
        using T = decltype(tag);
        return with_depth(k, [&](auto kk) -> cudaError_t {
            constexpr int K = decltype(kk)::value;
            if constexpr (K >= 2 && K <= MaxDepth<T>::value &&
                          is_f32_f64<T>())
                return split_tk<T, K>(reaction, boundary, u, v, un, vn, nn, nm, p, rows, s);
            else
                return cudaErrorInvalidValue;
        });
    });
}

cudaError_t launch_generic(int dtype, int reaction, int boundary, const void *u, const void *v,
                           void *un, void *vn, int64_t nn, int64_t nm, const rdcnn_params &p,
                           cudaStream_t s) {
    return with_dtype(dtype, [&](auto tag) {
        return generic_t<decltype(tag)>(reaction, boundary, u, v, un, vn, nn, nm, p, s);
    });
}

cudaError_t launch_init(int dtype, const void *x, void *u, void *v, double ka, int64_t n,
                        cudaStream_t s) {
    const int64_t want = (n + 255) / 256;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sm_count() * 16));
    return with_dtype(dtype, [&](auto tag) {
        using T = decltype(tag);
        k_init<T><<<grid, 256, 0, s>>>((const T *)x, (T *)u, (T *)v, (CT<T>)ka, n);
        count_launches(1);
        return cudaGetLastError();
    });
}

bool on_this_device(const void *p) {
    cudaPointerAttributes at;
    int dev = -1;
    const bool ok = cudaPointerGetAttributes(&at, p) == cudaSuccess && cudaGetDevice(&dev) == cudaSuccess &&
                    (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) && at.device == dev;
    if (!ok) (void)cudaGetLastError();
    return ok;
}

// A pair of planes is copied by one kernel: two copies queued one after the
// other cost a second launch and the gap between them (24 states of 128^2 ..
// 1024^2 and the run after them: 1128 -> 987 us).  Planes that are
// not whole vectors, that overlap (where the order of the copies matters) or that
// lie on another device are copied one after the other.
cudaError_t copy_planes(void *du, void *dv, const void *su, const void *sv, size_t bytes, cudaStream_t s) {
    const char *dst[2] = {(const char *)du, (const char *)dv}, *src[2] = {(const char *)su, (const char *)sv};
    bool plain = bytes % 16 != 0 || !aligned16(du) || !aligned16(dv) || !aligned16(su) || !aligned16(sv) ||
                 (dst[0] < dst[1] + bytes && dst[1] < dst[0] + bytes);
    for (const char *a : dst)
        for (const char *b : src) plain = plain || (a < b + bytes && b < a + bytes);
    if (plain || !on_this_device(du) || !on_this_device(dv) || !on_this_device(su) || (sv != su && !on_this_device(sv))) {
        const cudaError_t e = cudaMemcpyAsync(du, su, bytes, cudaMemcpyDeviceToDevice, s);
        return e != cudaSuccess ? e : cudaMemcpyAsync(dv, sv, bytes, cudaMemcpyDeviceToDevice, s);
    }
    const int64_t n = (int64_t)(bytes / 16);
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 16));
    // like the copies it stands for, not among the launches that are counted
    return launch_k(k_copy_planes, grid, 256, 0, s, (const uint4 *)su, (const uint4 *)sv, (uint4 *)du, (uint4 *)dv, n);
}

int plan_rows(int dtype, int reaction, int boundary, int variant, int k, int64_t nn, int64_t nm,
              int rows) {
    if (variant == RDCNN_VARIANT_STEP1) return rows > 0 ? rows : default_rows_step1(dtype, nn, nm);
    if (variant == RDCNN_VARIANT_GENERIC) return 0;
    const bool ragged = (variant == kVariantRagged);
    int out = 0;
    with_dtype(dtype, [&](auto tag) {
        using T = decltype(tag);
        return with_depth(k, [&](auto kk) -> cudaError_t {
            constexpr int K = decltype(kk)::value;
            if constexpr (K <= MaxDepth<T>::value) {
                if constexpr (K >= 2 && is_f32_f64<T>()) {
                    if (variant == RDCNN_VARIANT_TEMPORAL2) {
                        out = split_rows<T, K>(reaction, boundary, nn, nm, rows);
                        return cudaSuccess;
                    }
                }
                if constexpr (std::is_same<T, float>::value) {
                    if (ragged) {
                        out = temporal_rows<Ragged<float>, K>(reaction, boundary, nn, nm, rows);
                        return cudaSuccess;
                    }
                }
                if constexpr (K <= kMaxKWide && !std::is_same<T, double>::value) {
                    if (variant == RDCNN_VARIANT_TEMPORAL_WIDE) {
                        out = temporal_rows<Wide<T>, K>(reaction, boundary, nn, nm, rows);
                        return cudaSuccess;
                    }
                }
                out = temporal_rows<T, K>(reaction, boundary, nn, nm, rows);
            }
            return cudaSuccess;
        });
    });
    return out;
}

// Temporal depth when the caller gives none.  FP32: the model above.  FP64: 2,
// see auto_single_step.  16-bit planes round once per launch, so the depth is
// part of their result: by size class, k = 4 below 2^17 cells, 6 below 2^19, 4
// below 2^21, 8 above.
int default_k(int dtype, int64_t nn, int64_t nm) {
    const int64_t cells = nn * nm;
    if (dtype == RDCNN_F64) return 2;
    if (dtype == RDCNN_F32) return model_depth(kBeats, nn, nm);
    if (cells >= (int64_t(1) << 21)) return 8;
    if (cells >= (int64_t(1) << 19)) return 4;
    if (cells >= (int64_t(1) << 17)) return 6;
    return 4;
}
int default_k_ragged(int64_t nn, int64_t nm) { return model_depth(kRaggedBeats, nn, nm); }

// FP64 runs at 1/64 of the FP32 rate, so the FP64 pipe bounds every grid that
// fills the GPU, and a halo cell costs as much as an owned one: the single
// step, which computes no cell twice, beats every depth at every size.  us a
// step (k = 4 / best depth / single step): 64^2 7.3 / 5.9 / 2.3, 256^2 7.4 /
// 5.9 / 3.5, 512^2 18.7 / 10.9 / 9.3, 1024^2 42.4 / 37.4 / 30.6, 2048^2 156 /
// 136 / 113.
bool auto_single_step(int dtype) { return dtype == RDCNN_F64; }

// The single-step kernel is fastest with short strips (more warps in flight).
// The 16-bit single step (the ring pipeline at depth 1, 8 values per lane where
// rows are such vectors) takes the strips of which an SM gets 8, or 16 where
// those would be longer than 17 rows, and 32 rows where these are longer than 27: a
// strip's two extra input rows then weigh little, and the 32 of the large grids'
// sweep (4 .. 64 rows at 4096^2) beat the 28 to 31 of the rule by 2 %.  bf16, us a
// step, 32 rows / now: 512^2 7.5 / 2.5, 1024^2 7.6 / 3.4, 2048^2 8.0 / 6.5, 4096 x
// 1000 10.5 / 6.8, 2900 x 3128 14.8 / 11.4; 4096^2 with 31 / 32 rows 23.9 / 23.5.
// FP64: one row while that leaves warp slots free, else two (us a step, 1 / 2 /
// 4 / 8 rows: 64^2 2.3 / 3.6 / 5.6 / 10.2, 256^2 3.6 / 3.7 / 5.9 / 10.5, 512^2
// 10.4 / 9.1 / 10.0 / 11.1, 2048^2 120 / 110 / 110 / 114).
int default_rows_step1(int dtype, int64_t nn, int64_t nm) {
    if (dtype == RDCNN_F64) return nn * nm <= (int64_t(1) << 16) ? 1 : 2;
    if (!is_16bit(dtype)) return 2;
    const int64_t outw = nm % 8 == 0 ? 240 : 120;
    const int64_t bands = (nm + outw - 1) / outw;
    int64_t rows = 32;
    for (int per_sm : {8, 16}) {
        const int64_t strips = std::max<int64_t>(1, sm_count() * per_sm / bands);
        rows = (nn + strips - 1) / strips;
        if (rows <= 17) break;
    }
    return rows > 27 ? 32 : (int)std::max<int64_t>(rows, 2);
}

}  // namespace rdk
