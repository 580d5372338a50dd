// team.cu -- launch of the team kernel (team.cuh) for every size of
// at most 256 x 256.
#include "team.cuh"
#include "variants.cuh"

namespace admm {

namespace {

template <int H, int W, bool ANISO>
cudaError_t config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* at, int slots, cudaStream_t s) {
    using C = TeamCfg<H, W>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(tv_team<H, W, ANISO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)C::SMEM);
        if (e == cudaSuccess && C::DSM && C::C > 8)
            e = cudaFuncSetAttribute(tv_team<H, W, ANISO>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(C::C * slots);
    cfg->blockDim = dim3(C::NT);
    cfg->dynamicSmemBytes = C::SMEM;
    cfg->stream = s;
    if (C::DSM) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = C::C;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
    } else {
        at[0].id = cudaLaunchAttributeCooperative;   // the CTAs wait for one another
        at[0].val.cooperative = 1;
    }
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return cudaSuccess;
}

template <int H, int W, bool ANISO>
int capacity() {
    static int n = -1;
    if (n < 0) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at[1];
        int v = 0;
        cudaError_t e = config<H, W, ANISO>(&cfg, at, 1, nullptr);
        if (e == cudaSuccess && TeamCfg<H, W>::DSM) {
            e = cudaOccupancyMaxActiveClusters(&v, tv_team<H, W, ANISO>, &cfg);
        } else if (e == cudaSuccess) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, tv_team<H, W, ANISO>, TeamCfg<H, W>::NT,
                                                              TeamCfg<H, W>::SMEM);
            v = v * device_sm_count() / TeamCfg<H, W>::C;
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            v = 0;
        }
        n = v;
    }
    return n;
}

template <int H, int W, bool ANISO>
cudaError_t launch(const ProbDesc* d, SlotTable sl, int slots, int Wp, const float2* tw, int* n_active, int max_steps,
                   cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    cudaError_t e = config<H, W, ANISO>(&cfg, at, slots, s);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, tv_team<H, W, ANISO>, d, sl, Wp, tw, n_active, max_steps);
}

#define ADMM_TEAM_SIZES(X) \
    X(64, 64) X(64, 128) X(64, 256) X(128, 64) X(128, 128) X(128, 256) X(256, 64) X(256, 128) X(256, 256)

}  // namespace

int tv_team_capacity(int H, int W, bool aniso) {
#define ADMM_CASE(h, w) \
    if (H == h && W == w) return aniso ? capacity<h, w, true>() : capacity<h, w, false>();
    ADMM_TEAM_SIZES(ADMM_CASE)
#undef ADMM_CASE
    return 0;
}

bool tv_team_cluster(int H, int W) {
#define ADMM_CASE(h, w) \
    if (H == h && W == w) return TeamCfg<h, w>::DSM;
    ADMM_TEAM_SIZES(ADMM_CASE)
#undef ADMM_CASE
    return false;
}

cudaError_t launch_tv_team(int H, int W, bool aniso, const ProbDesc* d, SlotTable sl, int slots, int Wp,
                              const float2* tw, int* n_active, int max_steps, cudaStream_t s) {
#define ADMM_CASE(h, w)                                                                                     \
    if (H == h && W == w)                                                                                   \
        return aniso ? launch<h, w, true>(d, sl, slots, Wp, tw, n_active, max_steps, s)                     \
                     : launch<h, w, false>(d, sl, slots, Wp, tw, n_active, max_steps, s);
    ADMM_TEAM_SIZES(ADMM_CASE)
#undef ADMM_CASE
    return cudaErrorInvalidValue;
}

}  // namespace admm
