// umi_variants.h -- table of compiled kernel variants: lanes per window G,
// register slots per lane R, and MINB, the CTAs of 256 threads per SM the
// register allocation aims for.  Each variant serves windows with W <= G*R.
#pragma once

#include <cuda_runtime.h>

#include "umi_kernel.cuh"

namespace umi {

typedef cudaError_t (*LaunchFn)(const LaunchArgs &args, int grid, int threads, size_t smem,
                                cudaStream_t stream);

// Kernel flavours: index = kFlagDiag | kFlagMad | kFlagMin bits.
constexpr int kFlavours = 8;

struct Variant {
    int G;
    int R;
    int minb;
    LaunchFn launch[kFlavours];
    const void *kernel[kFlavours];  // for occupancy queries and attributes
};

// Launches a tile kernel so that it may be set up while the kernel before it
// in the stream ends (its griddepcontrol.wait holds it until that one's results
// are visible): between plain launches the GPU waits out whole steps of about
// 2 us.  One curve after another: W = 25 6.2 -> 5.4 us, W = 361 22.6 -> 20.0,
// W = 721 32.8 -> 30.3.  The kernels do not trigger the next launch early
// (griddepcontrol.launch_dependents): its CTAs would settle on the SMs that
// free up first, which left grids of less than a wave uneven (22.6 -> 27.5 us
// for one curve at W = 361 in chains of 6).
inline cudaError_t launch_dependent(void (*kernel)(LaunchArgs), const LaunchArgs &a, int grid, int threads,
                                    size_t smem, cudaStream_t st)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

// All compiled variants, ordered by slot capacity G*R (ascending).
const Variant *variant_table(int *count);

}  // namespace umi

// Defines the launchers of one (G, R, MINB) variant in the including translation unit.
#define UMI_VNAME(p, G_, R_, M_) p##G_##_##R_##_##M_
#define UMI_DEFINE_VARIANT(G_, R_, M_)                                                        \
    namespace umi {                                                                           \
    template <int F>                                                                          \
    static cudaError_t UMI_VNAME(launch_, G_, R_, M_)(const LaunchArgs &a, int grid,          \
                                                      int threads, size_t smem,               \
                                                      cudaStream_t st)                        \
    {                                                                                         \
        return launch_dependent(umi_tile_kernel<G_, R_, M_, F>, a, grid, threads, smem, st);  \
    }                                                                                         \
    template <int F>                                                                          \
    static void UMI_VNAME(fill_flavour_, G_, R_, M_)(Variant * v)                             \
    {                                                                                         \
        v->launch[F] = UMI_VNAME(launch_, G_, R_, M_)<F>;                                     \
        v->kernel[F] = (const void *)umi_tile_kernel<G_, R_, M_, F>;                          \
    }                                                                                         \
    void UMI_VNAME(fill_, G_, R_, M_)(Variant * v)                                            \
    {                                                                                         \
        v->G = G_;                                                                            \
        v->R = R_;                                                                            \
        v->minb = M_;                                                                         \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<0>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<1>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<2>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<3>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<4>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<5>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<6>(v);                                           \
        UMI_VNAME(fill_flavour_, G_, R_, M_)<7>(v);                                           \
    }                                                                                         \
    }

#define UMI_DECLARE_VARIANT(G_, R_, M_)                   \
    namespace umi {                                       \
    void UMI_VNAME(fill_, G_, R_, M_)(Variant * v);       \
    }

// The variant list: (G, R, MINB), ordered by slot capacity G*R; for equal
// capacity the first entry is the default and the autotuner may pick others.
// Every slot past W is work for nothing, so from 64 to 1,088 slots the capacities
// follow each other within about a fifth (3 to 21 %); below, with few slots, they
// step by 23 to 100 %, and from 1,088 to 1,536 (41 %) and 2,176 to 2,944 (35 %)
// there is none between.  A capacity is cut into as few lanes as 56 to 68
// slots allow: fewer lanes reduce in fewer steps and serve more windows per
// warp at the same 16 warps per SM.  ns per window, large bands: W = 73 (2,38)
// 0.106, (4,20) 0.120, (4,32) 0.176; W = 217 (4,56) 0.289, (8,28) 0.342, (8,46)
// 0.50; W = 433 (8,56) 0.602, (16,28) 0.653, (16,48) 1.05; W = 2521 (32,96) 4.2,
// (32,128) 5.4.  (2,32,2) and (4,32,2) are there because small bands take the
// largest register budget among the near capacities and would otherwise skip
// to the next one; no 32-lane capacity lies between 721 and 1442, where small
// bands of W = 721 would take it in place of (16,48,2) (latency_variant's "within
// 2W"), so windows of 1,089 to 1,441 samples run on 1,536 slots.
#define UMI_VARIANT_LIST(X) \
    X(1, 8, 4)           \
    X(1, 16, 4)          \
    X(1, 26, 4)          \
    X(1, 32, 3)          \
    X(1, 40, 3)          \
    X(1, 52, 2)          \
    X(2, 32, 3)          \
    X(2, 32, 2)          \
    X(2, 38, 2)          \
    X(2, 44, 2)          \
    X(2, 52, 2)          \
    X(2, 62, 2)          \
    X(4, 32, 3)          \
    X(4, 32, 2)          \
    X(4, 38, 2)          \
    X(4, 46, 2)          \
    X(8, 24, 3)          \
    X(4, 56, 2)          \
    X(4, 68, 2)          \
    X(8, 40, 2)          \
    X(8, 46, 2)          \
    X(8, 46, 3)          \
    X(8, 48, 2)          \
    X(16, 24, 4)         \
    X(32, 12, 4)         \
    X(8, 56, 2)          \
    X(8, 68, 2)          \
    X(16, 40, 2)         \
    X(16, 48, 2)         \
    X(16, 56, 2)         \
    X(16, 68, 2)         \
    X(32, 48, 2)         \
    X(32, 56, 2)         \
    X(32, 68, 2)         \
    X(32, 92, 1)         \
    X(32, 112, 1)        \
    X(32, 128, 1)
