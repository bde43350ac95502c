// resident.cu -- which runs the cluster-resident kernel (resident.cuh) takes,
// and in which shape.
#include <algorithm>

#include "resident_launch.cuh"

extern template RDK_RESIDENT_SIG(2);
extern template RDK_RESIDENT_SIG(4);
extern template RDK_RESIDENT_SIG(8);
extern template RDK_RESIDENT_SIG(12);

namespace rdk {

namespace {

// Lane width, blocks of the cluster and warps of a block; every warp has
// 1 .. kResRows rows.  V = 0: the grid does not fit.
struct ResShape {
    int V = 0, blocks = 0, warps = 0;
};

// Sixteen blocks whatever the size (us a step with 16 / 8 / 4 / 1 blocks: 64^2
// 0.25 / 0.25 / 0.32 / 0.57, 128^2 0.32 / 0.41 / 0.60 / -, 256^2 0.62 / 0.92 / - / -,
// with plain rows handed on), and as many rows a warp as leave one warp to each
// of an SM's four schedulers, at most four: 64^2 with 1 / 2 / 4 rows 0.20 / 0.22 /
// 0.26, 256^2 with 2 / 4 rows 0.52 / 0.49, 512 x 256 with 4 rows 0.75.
// Against the launches it stands for (k = 4 or 6, replayed as a graph), T = 1024,
// us: 16 x 256 805 -> 345, 64^2 857 -> 181, 1024 x 128 1187 -> 740, 512 x 256 1187 ->
// 763, 251 x 253 1412 -> 709 (short runs: resident_pays).
// 257 to 384 columns (12 a lane) only up to 256 rows: us a step, launches /
// resident: 64 x 384 0.79 / 0.39, 128 x 300 0.79 / 0.46, 256 x 260 0.80 / 0.68, but
// 300^2 0.82 / 1.03, 384^2 0.96 / 1.04.
ResShape resident_shape(int64_t nn, int64_t nm) {
    ResShape s;
    if (nm < 16 || nm > (nn <= 256 ? 384 : 256) || nn < 1) return s;
    const int V = nm <= 64 ? 2 : nm <= 128 ? 4 : nm <= 256 ? 8 : 12;
    const int most = V >= 8 ? ResWarps<8>::value : ResWarps<4>::value;
    const int blocks = (int)std::min<int64_t>(16, nn);
    const int64_t per_block = (nn + blocks - 1) / blocks;
    const int64_t rows = std::min<int64_t>(kResRows, (per_block + 3) / 4);
    // no more warps than rows
    const int64_t warps = std::min<int64_t>((per_block + rows - 1) / rows, nn / blocks);
    if (warps > most || (nn + blocks * warps - 1) / (blocks * warps) > kResRows) return s;
    s.V = V;
    s.blocks = blocks;
    s.warps = (int)warps;
    return s;
}

}  // namespace

bool resident_fits(int64_t nn, int64_t nm) { return resident_shape(nn, nm).V != 0; }

// A cluster reads and writes the planes with 16 SMs, strided by the lanes' width,
// which short runs of the larger grids do not earn back: us of a launch, a base of
// 2.2 and the cells, and per step 0.15 and what a scheduler's warps hold, within 15 %
// of 18 shapes measured; zero flux and overlapping last lanes cost more.  The
// other side is the launches it stands for, and either side the host's time: a
// run's call 6 us and each launch 2.9; between marks, which copy the state from
// here but are written by the launches themselves, only those.  us before the cluster /
// always the cluster / chosen: 512 x 256 8 steps 11.8 / 19.3 / 11.7, 400 x 256 8 steps
// 11.6 / 15.2 / 11.6, every step kept (a slot) 512 x 256 10.6 / 15.7 / 2.9, 256^2 10.7 / 9.9 / 2.9.
bool resident_pays(int boundary, int64_t nn, int64_t nm, int64_t steps, bool marks, bool ragged, int k) {
    const ResShape q = resident_shape(nn, nm);
    const int64_t nwarps = (int64_t)q.blocks * q.warps;
    const double base = 2.2 + 1e-4 * (double)(nn * nm) * (q.V == 2 ? 0.15 : q.V == 4 ? 0.29 : 0.78);
    const double held = (double)((nn + nwarps - 1) / nwarps * q.V * ((q.warps + 3) / 4));
    const double step = (0.15 + 0.0088 * held + (q.V == 12 ? 0.08 : 0.0) + (q.V != 2 && nm % 4 != 0 ? 0.15 : 0.0)) *
                        (boundary == RDCNN_BC_ZEROFLUX ? 1.2 : 1.0);
    const double cluster = base + step * (double)steps;
    if (!marks && cluster <= 0.6 * (double)steps) return true;  // no launches take less
    double us;
    const int64_t n = stretch_launches(ragged, nn, nm, steps, k, marks ? -1 : 0, &us);
    if (marks) return std::max(2 * kHostUs, cluster + 1.8) <= std::max((double)n * kHostUs, us);
    return std::max(6.0 + kHostUs, cluster) <= std::max(6.0 + (double)(n + n % 2) * kHostUs, us);  // odd: and a copy
}

cudaError_t launch_resident(int reaction, int boundary, void *u, void *v, int64_t nn, int64_t nm,
                            const rdcnn_params &p, int64_t steps, cudaStream_t s, bool give_up) {
    const ResShape q = resident_shape(nn, nm);
    auto go = [&](auto vv) {
        return resident_launch_v<decltype(vv)::value>(reaction, boundary, u, v, nn, nm, p, q.blocks, q.warps, steps,
                                                  give_up, s);
    };
    switch (q.V) {
        case 2: return go(IntC<2>{});
        case 4: return go(IntC<4>{});
        case 8: return go(IntC<8>{});
        case 12: return go(IntC<12>{});
        default: return cudaErrorNotSupported;
    }
}

}  // namespace rdk
