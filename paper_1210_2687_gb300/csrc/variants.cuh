// variants.cuh -- the kernel configurations the engine chooses between for a
// size class, and their launchers.
//
// Every side length has a short list of compiled configurations of the TV
// row phase (rows per strip R, walk rows in flight D, threads per CTA NT) and
// of the column phase (columns per CTA CB). Untuned classes take entry 0 of
// the column phase's list and the row configuration that tv_row_default
// names. The autotuner (admm_deconv_autotune) times the combinations on the
// device and records the fastest per (device, H, W, regulariser, levels);
// plans created afterwards use it. The instantiations are spread over
// several translation units (rows_small.cu, rows_512.cu, rows_large.cu,
// cols.cu) so that they compile in parallel.
#pragma once
#include <algorithm>

#include "kernels.cuh"

namespace admm {

using RowLaunchFn = cudaError_t (*)(const ProbDesc* d, SlotTable sl, int count, int H, int Wp, const float2* tw,
                                    int* n_active, cudaStream_t s);
using ColLaunchFn = cudaError_t (*)(const ProbDesc* d, SlotTable sl, int count, int Wc, int Wp, const float2* tw,
                                    cudaStream_t s);

struct RowVariant {
    int R, D, NT;
    RowLaunchFn fn;          // isotropic TV
    RowLaunchFn fn_aniso;    // anisotropic TV
};
struct ColVariant {
    int CB;
    int MB;   // CTAs per SM the registers are sized for (0: the default of the block)
    int persistent;   // 1: persistent CTAs with a double-buffered tile (col_phase_pers)
    ColLaunchFn fn;
};

// candidates for one side length (entry 0 = default); returns their number,
// 0 for an unsupported side
int tv_row_variants(int W, const RowVariant** out);
// The TV row configuration of an untuned class with `pixels` = H W problems
// in flight; every configuration gives the same bits. Short strips transform
// more halo rows, but their CTAs are many and small, which hides the walk's
// latencies: on narrow rows they always win, on rows of 512 only while a
// launch is short of CTAs; rows of 1024 take the longer strip as soon as
// their launches fill the GPU. Us per problem and iteration (both phases):
//   W   64  (16,4,256) -> (4,2,64)   64^2 x 256 0.40 -> 0.28, 512 x 64 x 1 22.8 -> 16.1
//   W  128  (16,4,256) -> (4,2,64)   128^2 x 64 0.87 -> 0.67, 512 x 128 x 4 6.46 -> 5.02
//   W  256  (8,4,256) -> (4,2,128)   256^2 x 64 1.74 -> 1.51, x 8 2.93 -> 2.83, 512 x 256 x 1 19.4 -> 18.5
//   W  512  (8,1,128) -> (4,1,128)   512^2 x 1 29.3 -> 23.7, x 4 9.08 -> 8.41, but x 8 6.63 -> 7.10, x 64 4.75 -> 5.06
//   W 1024  (4,2,256) -> (8,1,256)   1024^2 x 2 33.1 -> 31.8, x 8 25.9 -> 25.2, but x 1 40.3 -> 42.9
//   W 2048  (4,1,256) -> (2,1,256)   2048^2 x 1 152.8 -> 132.8, x 4 120.2 -> 115.3
inline int tv_row_default(int W, long long pixels) {
    const bool few = pixels <= 1ll << 20;
    switch (W) {
        case 64: return 3;
        case 128: return 3;
        case 256: return 4;
        case 512: return few ? 6 : 0;
        case 1024: return few ? 0 : 1;
        case 2048: return 2;
    }
    return 0;
}
int col_variants(int H, const ColVariant** out);

// per translation unit
int tv_row_variants_small(int W, const RowVariant** out);   // W = 64, 128, 256
int tv_row_variants_512(const RowVariant** out);            // W = 512
int tv_row_variants_large(int W, const RowVariant** out);   // W = 1024, 2048

template <int W, int R, int D, int NT, bool ANISO>
cudaError_t launch_row_tv_t(const ProbDesc* d, SlotTable sl, int count, int H, int Wp, const float2* tw,
                            int* n_active, cudaStream_t s) {
    static bool attr = false;
    const size_t smem = RowCfg<W, R, D, NT>::SMEM;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(row_phase_tv<W, R, D, NT, ANISO>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 grid(H / R, count);
    return launch_chain(row_phase_tv<W, R, D, NT, ANISO>, grid, dim3(NT), smem, s, d, sl, H, Wp, tw, n_active);
}

template <int H, int CB, int MB>
cudaError_t launch_col_t(const ProbDesc* d, SlotTable sl, int count, int Wc, int Wp, const float2* tw,
                         cudaStream_t s) {
    static bool attr = false;
    const size_t smem = ColCfg<H, CB>::SMEM;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(col_phase<H, CB, MB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    dim3 grid(Wp / CB, count);
    return launch_chain(col_phase<H, CB, MB>, grid, dim3(kThreads), smem, s, d, sl, Wc, Wp, tw);
}

// persistent column phase: three CTAs per SM (two tiles and the twiddles in
// shared memory) over the items of the launch
int device_sm_count();
template <int H, int CB>
cudaError_t launch_col_pers_t(const ProbDesc* d, SlotTable sl, int count, int Wc, int Wp, const float2* tw,
                              cudaStream_t s) {
    static bool attr = false;
    const size_t smem = (size_t)2 * H * CB * sizeof(float4) + (size_t)ColCfg<H, CB>::TWN * sizeof(float2);
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(col_phase_pers<H, CB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const int nblk = Wp / CB, nitems = nblk * count;
    const int grid = std::min(nitems, 3 * device_sm_count());
    if (grid <= 0) return cudaSuccess;
    return launch_chain(col_phase_pers<H, CB>, dim3(grid), dim3(kThreads), smem, s, d, sl, Wc, Wp, tw, nblk, nitems);
}

template <int W, int R, int D, int NT>
constexpr RowVariant row_variant() {
    return RowVariant{R, D, NT, &launch_row_tv_t<W, R, D, NT, false>, &launch_row_tv_t<W, R, D, NT, true>};
}
// MB > 0: registers sized for MB CTAs per SM instead of the default
template <int H, int CB, int MB = 0>
constexpr ColVariant col_variant() {
    return ColVariant{CB, MB, 0, &launch_col_t<H, CB, MB>};
}
template <int H>
constexpr ColVariant col_variant_pers() {
    return ColVariant{ColCfg<H, kThreads / (H / 8)>::G, 3, 1, &launch_col_pers_t<H, kThreads / (H / 8)>};
}

}  // namespace admm
