// resident_launch.cuh -- host launcher of k_resident for one lane width V; the
// resident_v*.cu units instantiate it, so the kernels of every model compile in
// parallel.
#pragma once

#include <atomic>

#include "internal.h"
#include "resident.cuh"

namespace rdk {

template <int V>
constexpr size_t resident_smem(int warps) {  // two parities x two directions x two fields, the mbarriers, the flag
    return (size_t)2 * warps * 2 * 2 * 128 * V + (size_t)16 * warps + 16;
}

// 16 where the current device can run a cluster of that many of the largest
// blocks (more than eight is the non-portable size, which not every partition of
// a GPU has room for), else 0: grids of sixteen rows and more are dealt to
// sixteen blocks.
template <int V, int RX, int BC, int RAG>
int resident_most() {
    auto *k = k_resident<V, RX, BC, RAG>;
    const int wmax = ResWarps<V>::value;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)resident_smem<V>(wmax)) == cudaSuccess &&
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = 16;
        cfg.blockDim = 32 * wmax;
        cfg.dynamicSmemBytes = resident_smem<V>(wmax);
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0) return 16;
    }
    (void)cudaGetLastError();
    return 0;
}

// Whether a cluster of `blocks` blocks of `warps` warps can run; asked once per device.
template <int V, int RX, int BC, int RAG>
bool resident_runs(int blocks, int warps) {
    static std::atomic<int> known[16];  // resident_most() + 1 by device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) return false;
    int most = known[dev].load(std::memory_order_acquire) - 1;
    if (most < 0) {
        most = resident_most<V, RX, BC, RAG>();
        known[dev].store(most + 1, std::memory_order_release);
    }
    return blocks <= most && warps <= ResWarps<V>::value;
}

// `steps` steps of (u, v) in place, or cudaErrorNotSupported with nothing launched.
template <int V>
cudaError_t resident_launch_v(int reaction, int boundary, void *u, void *v, int64_t nn, int64_t nm,
                              const rdcnn_params &p, int blocks, int warps, int64_t steps, bool give_up,
                              cudaStream_t s) {
    ResArgs a{(float *)u, (float *)v, (int)nn, (int)nm, (int)steps, blocks, warps, make_coef<float>(p, reaction),
              give_up ? kResGiveUpNs : kResWaitNs, give_up ? 1 : 0};
    return with_model(reaction, boundary, [&](auto rx, auto bc) -> cudaError_t {
        constexpr int RX = decltype(rx)::value;
        constexpr int BC = decltype(bc)::value;
        auto launch = [&](auto rag) -> cudaError_t {
            constexpr int RAG = decltype(rag)::value;
            if (!resident_runs<V, RX, BC, RAG>(blocks, warps)) return cudaErrorNotSupported;
            cudaLaunchAttribute at[2];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = blocks;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[1].val.programmaticStreamSerializationAllowed = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = blocks;
            cfg.blockDim = 32 * warps;
            cfg.dynamicSmemBytes = resident_smem<V>(warps);
            cfg.stream = s;
            cfg.attrs = at;
            cfg.numAttrs = pdl_enabled() ? 2 : 1;
            const cudaError_t e = cudaLaunchKernelEx(&cfg, k_resident<V, RX, BC, RAG>, (const ResArgs)a);
            count_launches(1);
            return e != cudaSuccess ? e : cudaGetLastError();
        };
        if (nm % V == 0) return launch(IntC<0>{});
        if constexpr (V > 8) {
            if (nm % 4 == 0) return launch(IntC<4>{});
        }
        return launch(IntC<1>{});
    });
}

}  // namespace rdk

#define RDK_RESIDENT_SIG(VV)                                                                                 \
    cudaError_t rdk::resident_launch_v<VV>(int, int, void *, void *, int64_t, int64_t, const rdcnn_params &, \
                                           int, int, int64_t, bool, cudaStream_t)
