// cnn.cu -- the learned warm start: a stack of 3 x 3 convolutions on BF16
// tensor cores (tcgen05.mma, FP32 accumulate in tensor memory), its backward
// pass and Adam. Not part of the paper; Theorem 1 (convergence from any u0,
// d0) is what lets a predicted start feed Algorithm 2.
//
// Layout. Activations and their gradients are BF16 in planes of eight
// channels: [image][C / 8][H][W][8], C padded to 8 (the network's input),
// 16 or 32. One plane row is
// W x 16 contiguous bytes, so a halo tile of a plane is a few long row
// segments (one TMA box of 160-byte rows for the tensor-core layers), and a
// pixel's eight channels are the 16-byte K slice the MMAs consume. The
// network's 4-channel output is FP32 [image][H][W][4]. Packed weights are
// BF16 [tap][cout][cin] (cin contiguous), the order in which the B operand of
// the MMA consumes them.
//
// Every convolution of the forward pass and every input gradient runs on
// tcgen05 (conv3x3_rows, and conv3x3_tc for the first layer and for widths that
// strips of 128 columns do not fit): the 32-channel layers with bias and ReLU,
// the input gradients gated by the ReLU of the layer below, and the last layer
// (4 outputs padded to 16) with bias into FP32.
//
// The weight gradients are contractions over pixels, also on tcgen05
// (conv3x3_wgrad_tc): both operands MN-major, straight from the same planes.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/admm_warmstart.h"

namespace admm {
bool alloc_fault_fire();   // ADMM_OPT_FAIL_ALLOC (engine.cu)
}

namespace {

using bf16 = __nv_bfloat16;

constexpr int kLayers = ADMM_CNN_LAYERS;
constexpr int kWidth = ADMM_CNN_WIDTH;
constexpr int kIn = 2, kOut = 4;
constexpr int kTile = 16;

// real (cout, cin) and padded channel counts of layer l
__host__ __device__ constexpr int layer_cin(int l) { return l == 0 ? kIn : kWidth; }
__host__ __device__ constexpr int layer_cout(int l) { return l == kLayers - 1 ? kOut : kWidth; }
constexpr int pad16(int c) { return c <= 16 ? 16 : 32; }
// the first layer's 2 input channels fill one plane of eight
constexpr int layer_cinp(int l) { return l == 0 ? 8 : pad16(layer_cin(l)); }
constexpr int layer_coutp(int l) { return l == kLayers - 1 ? 16 : kWidth; }

long long param_offset(int l) {
    long long o = 0;
    for (int j = 0; j < l; ++j) o += (long long)layer_cout(j) * layer_cin(j) * 9 + layer_cout(j);
    return o;
}
long long param_count() { return param_offset(kLayers); }

std::mutex g_cnn_mutex;
int g_cnn_test_stall = 0;            // ADMM_OPT_TEST_CNN_STALL: armed for the next pass (under g_cnn_mutex)
long long g_cnn_launches = 0;

int fail(cudaError_t) { return ADMM_ECUDA; }
#define CKC(call)                                  \
    do {                                           \
        cudaError_t e_ = (call);                   \
        if (e_ != cudaSuccess) return fail(e_);    \
    } while (0)

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// a + b of both FP32 halves
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t pair2(float lo, float hi) {
    return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
// one lane of the (converged) warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}\n" : "=r"(p));
    return p != 0;
}
// (lo, hi) rounded to BF16
__device__ __forceinline__ uint32_t cvt2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// max(., 0) of both BF16 halves (NaN gives 0, as fmaxf does)
__device__ __forceinline__ uint32_t relu2(uint32_t v) {
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0u));
    return r;
}
// all ones in each half whose BF16 value is > 0
__device__ __forceinline__ uint32_t positive2(uint32_t v) {
    uint32_t r;
    asm("set.gt.u32.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0u));
    return r;
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem));
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// ---------------------------------------------------------------------------
// network input: [M^T y, mask] in channels 0 and 1 of one plane of eight
// ---------------------------------------------------------------------------
__global__ void cnn_input_kernel(const float* __restrict__ ybar, const uint8_t* __restrict__ mask,
                                 bf16* __restrict__ a0, long long npx) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npx) return;
    const bool obs = mask[i] != 0;
    const float y = obs ? ybar[i] : 0.f;
    reinterpret_cast<uint4*>(a0)[i] =
        make_uint4(pack2(__float2bfloat16(y), __float2bfloat16(obs ? 1.f : 0.f)), 0u, 0u, 0u);
}

// epilogues of the convolutions
enum { kModeReluBf16 = 0, kModeOutF32 = 1, kModeGateBf16 = 2, kModeStart = 3 };

// planes of eight channels that a convolution's input has in memory: the output
// gradient's 4 channels are one plane, the second of its 16-channel operand zeros
__host__ __device__ constexpr int stored_planes(int cin) { return cin == 16 ? 1 : cin / 8; }

// Where the last layer writes a predicted start (kModeStart): x0 = s0 o0, d1 =
// s1 o1, d2 = (s2 o2, s2 o3) of image i to x0 + i hw and d0 + 3 i hw or, for
// separately stored problems (a batch solve's learned start), px0[i], pd0[i]
constexpr int kWsBatch = 16;
struct StartOut {
    float s0, s1, s2;
    int separate;
    int test_stall;              // test hook (ADMM_OPT_TEST_CNN_STALL): CTA 0 withholds an input row
    float* x0;
    float* d0;
    float* px0[kWsBatch];
    float* pd0[kWsBatch];
};

// ---------------------------------------------------------------------------
// 3 x 3 convolution on the fifth-generation tensor cores (tcgen05.mma,
// accumulator in tensor memory).
//
// A CTA of four warps walks output tiles of 8 x 16 pixels (M = 128, one
// accumulator row per pixel: tile row oy, column ox at M row 8 oy + ox), N =
// COUT output channels (32, or 16 for the last layer's 4 outputs), K = 9 taps
// x CIN input channels. Operands sit in shared
// memory in the no-swizzle K-major layout of 8-row x 16-byte core matrices:
//   A: the 10 x 18 halo tile as [CIN/8][180 halo pixels][8 channels]; the A
//      matrix of tap (dy, dx) starts at halo pixel 10 dy + dx, its 8-row
//      groups (one tile row each) are 10 pixels = 160 B apart and its K
//      chunks 180 x 16 B apart, so no im2col copy is needed;
//   B: the weights as [tap][CIN/8][COUT output channels][8].
// With one plane of input channels (CIN = 8, the first layer) the taps go in
// pairs, one per K = 16 MMA: the A descriptor's K-chunk offset is then the
// pixel distance from the pair's first tap to its second (5 MMAs per tile,
// the ninth tap paired with a zero weight slot).
// The halo tile arrives by one TMA copy (cp.async.bulk.tensor, a 4-D view of
// the eight-channel planes whose innermost dimension merges a plane row's
// columns and channels, so each box row is 10 pixels x 16 B = 160 contiguous
// bytes and the box lands in shared memory already in the A layout; rows and
// columns outside the image read as zero), double-buffered. One thread issues
// the 9 x CIN/16 MMAs of a tile (K = 16 each; 5 for CIN = 8) and commits them
// to an mbarrier; the four warps wait (bounded), read their 32 lanes of the
// accumulator (tcgen05.ld) and apply bias + ReLU (forward) or the ReLU gate of
// the layer below (input gradient), storing four BF16 planes, or bias alone
// into the network's FP32 output (last layer).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t sh_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
// offsets >> 4, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: F32 accumulator, BF16 A and B, both
// K-major, M = 128, N = n (a multiple of 16)
__host__ __device__ constexpr uint32_t idesc_m128(uint32_t n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

__device__ __forceinline__ void umma_f16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}

__device__ __forceinline__ unsigned long long gtimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for phase `parity` of the mbarrier, at most about a second. try_wait
// suspends the thread in hardware until the phase completes or the time limit
// given here (1 ms) passes, so the loop does not poll: a poll is a
// shared-memory access, and the tensor cores need that bandwidth. The clock is
// read only after a failed try: %globaltimer takes hundreds of cycles, and most
// waits find their phase complete.
__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity), "r"(1000000u)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t parity) {
    if (mbar_try(mbar, parity)) return true;
    const unsigned long long t0 = gtimer_ns();
    do {
        if (mbar_try(mbar, parity)) return true;
    } while (gtimer_ns() - t0 <= 1000000000ull);
    return false;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 32 consecutive FP32 columns of this thread's accumulator lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 8 or 16 consecutive FP32 columns of this thread's accumulator lane
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[8]) {
    uint32_t r[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// clear N (16 or 32) consecutive columns of this warp's accumulator lanes
template <int N>
__device__ __forceinline__ void tmem_zero(uint32_t taddr) {
    static_assert(N == 16 || N == 32, "columns");
    if constexpr (N == 32)
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,"
            "%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n\ttcgen05.wait::st.sync.aligned;\n" ::"r"(taddr),
            "r"(0u)
            : "memory");
    else
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};\n\t"
            "tcgen05.wait::st.sync.aligned;\n" ::"r"(taddr),
            "r"(0u)
            : "memory");
}

// Programmatic dependent launch of the network's layers. A layer's CTAs are all
// resident (the grids are persistent), so each releases its successor as soon
// as it holds its tensor memory (layer_release): the successor's CTAs take the
// place of CTAs that end, load their weights and set up while the last ones
// still run, and wait for the predecessor's completion before they touch
// activations (layer_wait). The release comes after the tensor-memory
// allocation, so a waiting successor never holds what a predecessor still
// needs. Weights may be read before the wait: the chain's first launch is a
// plain one, after everything that wrote them. Both are no-ops in a plain launch.
// Predicted starts of 16 x 512^2: 873 -> 777 us; loss and gradients of 16 x 256^2: 1019 -> 902 us.
__device__ __forceinline__ void layer_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void layer_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The network's error state. A kernel whose bounded wait ran out sets `flag`
// (device) and *host (pinned), which the next call on the network sees without
// waiting; parameter updates are left out while the flag is set, and counted.
struct NetErr {
    int flag, skipped;
    int* host;
};
__device__ __forceinline__ void net_fail(NetErr* e) {
    atomicExch(&e->flag, 1);
    *static_cast<volatile int*>(e->host) = 1;
    __threadfence_system();
}

constexpr int kTcTW = 8, kTcTH = 16;                 // output tile (M = 128)
constexpr int kTcHW = kTcTW + 2, kTcHH = kTcTH + 2;  // halo tile
constexpr int kTcNP = kTcHW * kTcHH;                 // 180 halo pixels

// tin: TMA view of the input [img][CIN / 8][H][W][8] (see conv_tc); wpk:
// [9][COUT][CIN]; MODE kModeReluBf16 (bias, ReLU; out bf16 [img][4][H][W][8]),
// kModeGateBf16 (gate and out bf16 [img][4][H][W][8]) or kModeOutF32 (bias of
// the 4 outputs; out float [img][H][W][4]); err: told if a wait ran out (the CTA then stops,
// after a bounded wait for its own copies and MMAs still in flight).
//
// Pipeline of the CTA's i-th tile (halo buffer and accumulator i & 1): thread
// 0 waits for the halo of tile i + 1 and issues its MMAs into the other
// accumulator; all four warps then wait for tile i's MMAs, thread 0 starts the
// copy of tile i + 2's halo into the buffer they have finished reading, and
// the warps read tile i's accumulator and store it while the tensor cores work
// on tile i + 1.
template <int CIN, int MODE>
__global__ void __launch_bounds__(128)
conv3x3_tc(const __grid_constant__ CUtensorMap tin, const bf16* __restrict__ wpk, const float* __restrict__ bias,
           void* __restrict__ out, const bf16* __restrict__ gate, int H, int W, int count, NetErr* __restrict__ err) {
    constexpr int COUT = MODE == kModeOutF32 ? 16 : 32, CH = CIN / 8;
    constexpr int BOXBYTES = CH * kTcNP * 16;                  // one halo box
    constexpr int ABYTES = (BOXBYTES + 127) / 128 * 128;        // (each halo buffer on a 128-byte boundary)
    constexpr uint32_t kTmemCols = 2 * COUT;   // two accumulators
    // weight slots: the 9 taps, or with one plane of input channels (CIN = 8)
    // taps 0..7, a zero slot and tap 8, so that the MMAs take the taps in
    // pairs (0,1) (2,3) (4,5) (6,7) (zero,8), one per K = 16
    constexpr int NSLOT = CIN == 8 ? 10 : 9;
    static_assert(CIN == 8 || CIN == 16 || CIN == 32, "input channels");
    __shared__ __align__(128) unsigned char smA[2][ABYTES];
    __shared__ __align__(128) unsigned char smW[NSLOT * CH * COUT * 16];
    __shared__ float smB[32];
    // 0, 1: halo of buffer 0 / 1 landed; 2, 3: MMAs into accumulator 0 / 1 done
    __shared__ __align__(8) unsigned long long bars[4];
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    for (int e = tid; e < NSLOT * COUT * CH; e += 128) {
        const int sc = e / CH, k = e - sc * CH;       // sc = slot * COUT + output channel
        const int slot = sc / COUT, co = sc - slot * COUT;
        const int tap = CIN == 8 ? (slot < 8 ? slot : (slot == 9 ? 8 : -1)) : slot;
        unsigned char* dst = smW + ((slot * CH + k) * COUT + co) * 16;
        if (tap >= 0)
            cp_async16(dst, wpk + ((size_t)tap * COUT + co) * CIN + k * 8);
        else
            *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
    }
    if ((MODE == kModeReluBf16 && tid < COUT) || (MODE == kModeOutF32 && tid < kOut)) smB[tid] = bias[tid];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sh_addr(&tmem_base)),
                     "n"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const int tiles_x = W / kTcTW, per_img = tiles_x * (H / kTcTH);
    const int ntiles = per_img * count, G = gridDim.x;
    const uint64_t tmap = reinterpret_cast<uint64_t>(&tin);
    // phase bits (bit b: barrier of buffer / accumulator b) and, in thread 0,
    // the copies and MMA groups issued but not yet seen complete
    uint32_t hph = 0, mph = 0, pend_h = 0, pend_m = 0;
    // one TMA copy of tile t's halo into buffer b (thread 0)
    auto issue = [&](int t, int b) {
        const int img = t / per_img, rem = t - img * per_img;
        const int y0 = (rem / tiles_x) * kTcTH, x0 = (rem % tiles_x) * kTcTW;
        const uint32_t bar = sh_addr(&bars[b]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(BOXBYTES) : "memory");
        // x: element (column x0 - 1, channel 0) of the merged row, a multiple of 8
        // elements (16 B); column -1 and columns past W - 1 read as zero
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
            "%5}], [%6];" ::"r"(sh_addr(smA[b])),
            "l"(tmap), "r"((x0 - 1) * 8), "r"(y0 - 1), "r"(0), "r"(img), "r"(bar)
            : "memory");
        pend_h |= 1u << b;
    };
    if (tid == 0) {
        for (int i = 0; i < 4; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sh_addr(&bars[i])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
        layer_wait();
        if ((int)blockIdx.x < ntiles) issue(blockIdx.x, 0);
        if ((int)blockIdx.x + G < ntiles) issue(blockIdx.x + G, 1);
    }
    layer_wait();
    cp_async_wait_all();
    fence_async_shared();        // the weights (generic proxy) are visible to the tensor cores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    layer_release();
    const uint32_t tmem = tmem_base;
    const uint32_t wBase = sh_addr(smW);
    // thread 0: wait for the halo in buffer b, then issue the tile's MMAs into
    // accumulator b (columns COUT b) and commit them to bars[2 + b]
    auto mma_tile = [&](int b) -> bool {
        if (!mbar_wait_bounded(sh_addr(&bars[b]), (hph >> b) & 1u)) return false;
        hph ^= 1u << b;
        pend_h &= ~(1u << b);
        tc_fence_after();
        const uint32_t aBase = sh_addr(smA[b]), d = tmem + (uint32_t)COUT * b;
        if constexpr (CIN == 8) {
            // K chunk 0 of pair j is tap a (or the zero slot), chunk 1 tap b: the
            // A descriptor starts at tap a's halo pixel and steps to tap b's by
            // its K-chunk offset (halo pixel of a tap (dy, dx): 10 dy + dx)
            constexpr int pa[5] = {0, 2, 11, 20, 21};   // chunk 0: taps 0, 2, 4, 6; any pixel for the zero slot
            constexpr int pd[5] = {1, 8, 1, 1, 1};      // chunk 1: taps 1, 3, 5, 7, 8
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                const uint64_t a = umma_desc(aBase + pa[j] * 16, pd[j] * 16, kTcHW * 16);
                const uint64_t bd = umma_desc(wBase + 2 * j * COUT * 16, COUT * 16, 8 * 16);
                umma_f16(d, a, bd, idesc_m128(COUT), j != 0 ? 1u : 0u);
            }
        } else {
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int dy = tap / 3, dx = tap - 3 * (tap / 3);
#pragma unroll
                for (int j = 0; j < CH / 2; ++j) {
                    const uint64_t a =
                        umma_desc(aBase + (2 * j * kTcNP + dy * kTcHW + dx) * 16, kTcNP * 16, kTcHW * 16);
                    const uint64_t bd = umma_desc(wBase + (tap * CH + 2 * j) * COUT * 16, COUT * 16, 8 * 16);
                    umma_f16(d, a, bd, idesc_m128(COUT), (tap | j) != 0 ? 1u : 0u);
                }
            }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         sh_addr(&bars[2 + b]))
                     : "memory");
        pend_m |= 1u << b;
        return true;
    };
    bool ok = true;
    if (tid == 0 && (int)blockIdx.x < ntiles) ok = mma_tile(0);
    int it = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += G, ++it) {
        const int b = it & 1;
        // accumulator b ^ 1 was last read by the previous tile's epilogue,
        // which ended at the block barrier below
        if (tid == 0 && ok && tile + G < ntiles) ok = mma_tile(b ^ 1);
        const bool got = mbar_wait_bounded(sh_addr(&bars[2 + b]), (mph >> b) & 1u);
        if (got) {
            mph ^= 1u << b;
            pend_m &= ~(1u << b);
        }
        ok = __syncthreads_and(got && ok) != 0;
        if (!ok) break;
        // tile's MMAs are complete, so its halo buffer is free
        if (tid == 0 && tile + 2 * G < ntiles) issue(tile + 2 * G, b);
        tc_fence_after();
        const int img = tile / per_img, rem = tile - img * per_img;
        const int y0 = (rem / tiles_x) * kTcTH, x0 = (rem % tiles_x) * kTcTW;
        const int oy = 4 * warp + (lane >> 3), ox = lane & 7;
        const size_t hw = (size_t)H * W;
        const uint32_t tacc = tmem + (uint32_t)COUT * b + ((uint32_t)(32 * warp) << 16);
        if constexpr (MODE == kModeOutF32) {
            float v[16];
            tmem_ld(tacc, v);
            const size_t px = (size_t)img * hw + (size_t)(y0 + oy) * W + (x0 + ox);
            reinterpret_cast<float4*>(out)[px] =
                make_float4(v[0] + smB[0], v[1] + smB[1], v[2] + smB[2], v[3] + smB[3]);
        } else {
            float v[32];
            tmem_ld32(tacc, v);
            // pixel's slot in plane 0 of its image; plane q is q hw slots further
            const size_t px = (size_t)img * 4 * hw + (size_t)(y0 + oy) * W + (x0 + ox);
            uint32_t pk[16];
            if (MODE == kModeReluBf16) {
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    pk[c] = pack2(__float2bfloat16(fmaxf(v[2 * c] + smB[2 * c], 0.f)),
                                  __float2bfloat16(fmaxf(v[2 * c + 1] + smB[2 * c + 1], 0.f)));
            } else {
                const uint4* gp = reinterpret_cast<const uint4*>(gate) + px;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 gv = gp[q * hw];
                    const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        const int c = 8 * q + 2 * h;
                        const float g0 = __bfloat162float(__ushort_as_bfloat16((unsigned short)(gw[h] & 0xFFFFu)));
                        const float g1 = __bfloat162float(__ushort_as_bfloat16((unsigned short)(gw[h] >> 16)));
                        pk[4 * q + h] = pack2(__float2bfloat16(g0 > 0.f ? v[c] : 0.f),
                                              __float2bfloat16(g1 > 0.f ? v[c + 1] : 0.f));
                    }
                }
            }
            uint4* op = reinterpret_cast<uint4*>(out) + px;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                op[q * hw] = make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
        }
        tc_fence_before();
        __syncthreads();             // accumulator b is free for tile + 2 G's MMAs
    }
    if (!ok && tid == 0) {
        net_fail(err);
        // let this CTA's own copies and MMAs still in flight finish (bounded)
        // before its tensor memory is released
        for (int b = 0; b < 2; ++b) {
            if (pend_h & (1u << b)) mbar_wait_bounded(sh_addr(&bars[b]), (hph >> b) & 1u);
            if (pend_m & (1u << b)) mbar_wait_bounded(sh_addr(&bars[2 + b]), (mph >> b) & 1u);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmemCols) : "memory");
}

// ---------------------------------------------------------------------------
// 3 x 3 convolution of 16 or 32 input channels, streaming down the image
//
// A CTA walks rows of a strip of 128 columns (M = 128, accumulator row =
// column). An input row is the A operand of three output rows at once: the
// accumulators of output rows r - 1, r, r + 1 are three slots of COUT columns
// in tensor memory (slot = row mod 3), and one MMA of N = 3 COUT adds input row
// r's products with the weights of dy = 2, 1, 0 to them. The weight blocks lie
// in the cyclic order dy = 2 1 0 2 1, so each of the three rotations of the
// slots is a window of three consecutive blocks. That is 6 MMAs (dx, half of
// the channels) per row of 128 pixels and 7 KB of shared-memory operand reads
// each, 2.6 cycles per pixel and SM where one 128 x 32 MMA per tap reads 5.6
// (conv3x3_tc): the layer is then bound by its HBM traffic (64 B in and out per
// pixel, 5.6 cycles), with no column halo in it and two halo rows per segment.
// Every output sees its products in the order (dy, dx, channels) of
// conv3x3_tc, so the results have the same bits.
//
// Work: the count x strips x H strip rows are cut into equal ranges, one per
// CTA (three CTAs per SM), each a segment or two of consecutive rows of one
// strip. Warp 0 copies input rows (cp.async.bulk, one per plane of eight
// channels) kRowStages ahead and writes the zeros outside the image; lane 0 of
// warp 1 issues the MMAs; warps 2..5 read a finished accumulator, clear its
// slot for the row that takes it over, and store the row: bias + ReLU or the
// ReLU gate of the layer below into BF16 planes, or bias into FP32 outputs.
// While a CTA's MMAs wait for a slot to be read, the other CTAs' run.
// Hidden layer at 16 x 512^2: 103 us (5.2 TB/s of activations), 126 us as
// 8 x 16 tiles; the last layer 72 against 95 us.
// ---------------------------------------------------------------------------
constexpr int kStrip = 128, kRowPx = kStrip + 2, kRowStages = 4;

template <int CIN, int MODE>
struct RowsCfg {
    static constexpr int CH = CIN / 8, COUT = MODE == kModeOutF32 || MODE == kModeStart ? 16 : 32;
    static constexpr int PL = stored_planes(CIN);
    static constexpr int STAGE = (CH * kRowPx * 16 + 127) / 128 * 128;   // one input row with its two halo columns
    static constexpr int WBLK = 2 * 5 * COUT * 16;                       // weights of one (dx, channel half): 5 blocks
    static constexpr int NWB = 3 * (CIN / 16);
    static constexpr int N = 3 * COUT;
    static constexpr int TMEM_COLS = N <= 64 ? 64 : 128;
    static constexpr size_t SMEM = (size_t)kRowStages * STAGE + (size_t)NWB * WBLK + 128;
    static constexpr int CTAS = 3;                                       // per SM
};

template <int CIN, int MODE>
__global__ void __launch_bounds__(192, 3)
conv3x3_rows(const bf16* __restrict__ in, const bf16* __restrict__ wpk, const float* __restrict__ bias,
             void* __restrict__ out, const bf16* __restrict__ gate, int H, int W, int count, NetErr* __restrict__ err,
             const __grid_constant__ StartOut st) {
    using C = RowsCfg<CIN, MODE>;
    constexpr int COUT = C::COUT, PL = C::PL, S = kRowStages;
    extern __shared__ unsigned char rows_raw[];
    __shared__ __align__(8) unsigned long long full[S], empty[S], acc_full[3], acc_empty[3], done;
    __shared__ __align__(16) float smB[32];
    __shared__ uint32_t tmem_base;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* sm = rows_raw + ((128u - (sh_addr(rows_raw) & 127u)) & 127u);
    unsigned char* smW = sm + S * C::STAGE;
    // weights [dx][channel half][8-channel chunk][block, output channel][8]
    for (int e = tid; e < C::NWB * 2 * 5 * COUT; e += 192) {
        const int n = e % (5 * COUT), kh = (e / (5 * COUT)) % 2, blk = e / (10 * COUT);
        const int dx = blk / (CIN / 16), j = blk % (CIN / 16), co = n % COUT;
        const int dy = (5 - n / COUT) % 3;            // blocks 0..4: 2 1 0 2 1
        cp_async16(smW + (size_t)e * 16, wpk + ((size_t)(dy * 3 + dx) * COUT + co) * CIN + (2 * j + kh) * 8);
    }
    if (MODE != kModeGateBf16 && tid < (COUT == 16 ? kOut : COUT)) smB[tid] = bias[tid];
    if constexpr (PL < C::CH) {
        // planes that are not in memory stay zero
        for (int e = tid; e < S * (C::CH - PL) * kRowPx; e += 192) {
            const int i = e / ((C::CH - PL) * kRowPx), k = e - i * ((C::CH - PL) * kRowPx);
            *reinterpret_cast<uint4*>(sm + i * C::STAGE + (PL * kRowPx + k) * 16) = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sh_addr(&tmem_base)),
                     "n"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    auto bar_init = [](unsigned long long* b, uint32_t n) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sh_addr(b)), "r"(n) : "memory");
    };
    auto arrive = [](unsigned long long* b) {
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sh_addr(b)) : "memory");
    };
    auto commit = [](unsigned long long* b) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sh_addr(b))
                     : "memory");
    };
    if (tid == 0) {
        for (int i = 0; i < S; ++i) {
            bar_init(&full[i], 1);
            bar_init(&empty[i], 1);
        }
        for (int i = 0; i < 3; ++i) {
            bar_init(&acc_full[i], 1);
            bar_init(&acc_empty[i], 4);
        }
        bar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cp_async_wait_all();
    fence_async_shared();        // the weights (generic proxy) are visible to the tensor cores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    layer_release();
    layer_wait();
    const uint32_t tmem = tmem_base;
    const int strips = (W + kStrip - 1) / kStrip;
    const long long total = (long long)count * strips * H;
    const long long a0 = total * blockIdx.x / gridDim.x, a1 = total * (blockIdx.x + 1) / gridDim.x;
    const size_t hw = (size_t)H * W;
    bool ok = true;
    int asked = 0, used = 0;     // input rows requested; released by the MMAs (producer)
    if (warp == 0) {
        int n = 0;
        for (long long pos = a0; pos < a1 && ok;) {
            const int col = (int)(pos / H), y0 = (int)(pos - (long long)col * H);
            const int R = (int)min((long long)(H - y0), a1 - pos);
            const int img = col / strips, xs = (col - img * strips) * kStrip;
            pos += R;
            const int c0 = max(xs - 1, 0), c1 = min(xs + kStrip + 1, W);
            const int lo = c0 - (xs - 1), hi = c1 - (xs - 1);          // slots [lo, hi) hold image columns
            for (int i = 0; i < R + 2; ++i, ++n) {
                const int s = n % S, r = y0 - 1 + i;
                if (n >= S) {
                    ok = mbar_wait_bounded(sh_addr(&empty[s]), (uint32_t)((n / S - 1) & 1));
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    used = n - S + 1;
                }
                unsigned char* sg = sm + s * C::STAGE;
                const bool inside = r >= 0 && r < H;
                const int h0 = inside ? lo : kRowPx, nz = kRowPx - (inside ? hi - lo : 0);
                if (nz > 0) {
                    // zeros outside the image: slots [0, h0) and, for a row inside, [hi, kRowPx)
                    for (int e = lane; e < nz * PL; e += 32) {
                        const int pl = e / nz, k = e - pl * nz;
                        const int slot = k < h0 ? k : hi + (k - h0);
                        *reinterpret_cast<uint4*>(sg + (pl * kRowPx + slot) * 16) = make_uint4(0u, 0u, 0u, 0u);
                    }
                    fence_async_shared();
                    __syncwarp();
                }
                if (lane == 0 && !(st.test_stall && blockIdx.x == 0 && n == 1)) {
                    const uint32_t bar = sh_addr(&full[s]);
                    if (inside) {
                        const uint32_t bytes = (uint32_t)(hi - lo) * 16u;
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes * PL)
                                     : "memory");
                        // read once here: what stays in L2 is the output, which the next layer reads
                        // (at 16 x 256^2, where it fits, 834 -> 807 us for loss and gradients)
                        uint64_t once;
                        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(once));
                        const bf16* src = in + ((size_t)img * PL * hw + (size_t)r * W + c0) * 8;
                        for (int pl = 0; pl < PL; ++pl)
                            asm volatile(
                                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, "
                                "[%3], %4;" ::"r"(
                                    sh_addr(sg + (pl * kRowPx + lo) * 16)),
                                "l"(src + (size_t)pl * hw * 8), "r"(bytes), "r"(bar), "l"(once)
                                : "memory");
                    } else {
                        arrive(&full[s]);
                    }
                }
                asked = n + 1;
            }
        }
        // every stage's last release has arrived before the CTA ends
        for (int k = max(0, n - S); ok && k < n; ++k)
            ok = mbar_wait_bounded(sh_addr(&empty[k % S]), (uint32_t)((k / S) & 1));
    } else if (warp == 1) {
        // The warp stays converged and one lane is elected around the issue
        // itself, so that the descriptors are uniform values; their start
        // address is the lowest field, in units of 16 bytes.
        const uint64_t a_in = umma_desc(sh_addr(sm), kRowPx * 16, 128);
        const uint64_t b_in = umma_desc(sh_addr(smW), 5 * COUT * 16, 128);
        uint32_t s = 0, fp = 0, eph = 0, need = 7;   // stage and phase; slots whose clearing is not yet seen (at first: all)
        auto slot_clear = [&](uint32_t k) -> bool {
            if (!((need >> k) & 1u)) return true;
            if (!mbar_wait_bounded(sh_addr(&acc_empty[k]), (eph >> k) & 1u)) return false;
            eph ^= 1u << k;
            need &= ~(1u << k);
            return true;
        };
        // one input row in the rotation PH of the slots
        auto row = [&](auto rotation, bool first, bool last) -> bool {
            constexpr int PH = decltype(rotation)::value, UP = (PH + 1) % 3, DOWN = (PH + 2) % 3;   // slots of rows r + 1, r - 1
            const bool go = mbar_wait_bounded(sh_addr(&full[s]), fp) && slot_clear(UP) &&
                            (!first || (slot_clear(PH) && slot_clear(DOWN)));
            // one answer for the warp: where the limit passes as the phase completes,
            // some lanes see it and some do not
            if (!__all_sync(0xffffffffu, go)) return false;
            tc_fence_after();
            const uint64_t a0 = a_in + s * (C::STAGE / 16);
            const uint64_t b0 = b_in + (PH == 0 ? 1 : (PH == 1 ? 0 : 2)) * COUT;         // window start
            if (elect_one()) {
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                    for (int j = 0; j < CIN / 16; ++j)
                        umma_f16(tmem, a0 + (2 * j * kRowPx + dx), b0 + (dx * (CIN / 16) + j) * (C::WBLK / 16),
                                 idesc_m128(C::N), 1u);
                }
                commit(&acc_full[DOWN]);             // output row r - 1 is complete
                commit(&empty[s]);
                if (last) {
                    // the two rows that the segment's last input row has begun are dropped
                    commit(&acc_full[PH]);
                    commit(&acc_full[UP]);
                }
            }
            __syncwarp();
            need |= last ? 7u : 1u << DOWN;
            if (++s == S) {
                s = 0;
                fp ^= 1u;
            }
            return true;
        };
        for (long long pos = a0; pos < a1 && ok;) {
            const int y0 = (int)(pos % H);
            const int R = (int)min((long long)(H - y0), a1 - pos);
            pos += R;
            // (every segment starts in rotation 0)
            const int n = R + 2;
            for (int t = 0; t < n && ok; t += 3) {
                ok = row(std::integral_constant<int, 0>(), t == 0, t + 1 == n);
                if (ok && t + 1 < n) ok = row(std::integral_constant<int, 1>(), false, t + 2 == n);
                if (ok && t + 2 < n) ok = row(std::integral_constant<int, 2>(), false, t + 3 == n);
            }
        }
        ok = __all_sync(0xffffffffu, ok);
        if (elect_one()) commit(&done);              // (the thread that has issued the MMAs)
    } else if (warp >= 2) {
        const int q = warp & 3;                      // this warp's quarter of the tensor-memory lanes
        const uint32_t tw = tmem + ((uint32_t)(32 * q) << 16);
        // clear slot k and hand it to the MMAs
        auto release = [&](int k) {
            tmem_zero<COUT>(tw + (uint32_t)(COUT * k));
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive(&acc_empty[k]);
        };
        for (int k = 0; k < 3; ++k) release(k);
        uint64_t bs[COUT / 2];                       // bias pairs
        if constexpr (MODE == kModeReluBf16) {
#pragma unroll
            for (int h = 0; h < COUT / 2; ++h) bs[h] = pair2(smB[2 * h], smB[2 * h + 1]);
        }
        uint32_t fph = 0;
        for (long long pos = a0; pos < a1 && ok;) {
            const int col = (int)(pos / H), y0 = (int)(pos - (long long)col * H);
            const int R = (int)min((long long)(H - y0), a1 - pos);
            const int img = col / strips, xs = (col - img * strips) * kStrip;
            pos += R;
            const int c = xs + 32 * q + lane;
            int k = 2;                               // slot of the drain: (d + 2) mod 3
            for (int d = 0; d < R + 4; ++d, k = k == 2 ? 0 : k + 1) {
                const int o = y0 - 2 + d;
                const bool keep = d >= 2 && d < R + 2 && c < W;
                // pixel's slot in plane 0 of its image; plane p is p hw slots further
                const size_t px = (size_t)img * (COUT == 16 ? 1 : 4) * hw + (size_t)o * W + c;
                uint4 gv[4];
                if constexpr (MODE == kModeGateBf16) {
                    const uint4* gp = reinterpret_cast<const uint4*>(gate) + px;
#pragma unroll
                    for (int p = 0; p < 4; ++p) gv[p] = keep ? __ldcs(gp + p * hw) : make_uint4(0u, 0u, 0u, 0u);
                }
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(sh_addr(&acc_full[k]), (fph >> k) & 1u));
                if (!ok) break;
                fph ^= 1u << k;
                tc_fence_after();
                float v[COUT];
                if constexpr (COUT == 32) tmem_ld32(tw + (uint32_t)(COUT * k), v);
                else tmem_ld(tw + (uint32_t)(COUT * k), v);
                release(k);
                if (!keep) continue;
                if constexpr (MODE == kModeOutF32) {
                    reinterpret_cast<float4*>(out)[px] =
                        make_float4(v[0] + smB[0], v[1] + smB[1], v[2] + smB[2], v[3] + smB[3]);
                } else if constexpr (MODE == kModeStart) {
                    const size_t ip = (size_t)o * W + c;
                    float* x0 = st.separate ? st.px0[img] : st.x0 + (size_t)img * hw;
                    float* d0 = st.separate ? st.pd0[img] : st.d0 + (size_t)img * 3 * hw;
                    x0[ip] = st.s0 * (v[0] + smB[0]);
                    d0[ip] = st.s1 * (v[1] + smB[1]);
                    reinterpret_cast<float2*>(d0 + hw)[ip] = make_float2(st.s2 * (v[2] + smB[2]), st.s2 * (v[3] + smB[3]));
                } else {
                    uint4* op = reinterpret_cast<uint4*>(out) + px;
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        uint32_t pk[4];
                        if constexpr (MODE == kModeReluBf16) {
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                const uint64_t u = add2(pair2(v[8 * p + 2 * h], v[8 * p + 2 * h + 1]), bs[4 * p + h]);
                                pk[h] = relu2(cvt2(__uint_as_float((uint32_t)u), __uint_as_float((uint32_t)(u >> 32))));
                            }
                        } else {
                            const uint32_t gw[4] = {gv[p].x, gv[p].y, gv[p].z, gv[p].w};
#pragma unroll
                            for (int h = 0; h < 4; ++h)
                                pk[h] = cvt2(v[8 * p + 2 * h], v[8 * p + 2 * h + 1]) & positive2(gw[h]);
                        }
                        op[p * hw] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                }
            }
        }
    }
    __syncwarp();
    ok = __syncthreads_and(ok) != 0;
    // every MMA issued is complete
    ok = __syncthreads_and(mbar_wait_bounded(sh_addr(&done), 0u) && ok) != 0;
    if (!ok && tid == 0) {
        // a wait ran out: let the copies still in flight land (bounded) before leaving
        net_fail(err);
        for (int k = max(used, asked - S); k < asked; ++k)
            mbar_wait_bounded(sh_addr(&full[k % S]), (uint32_t)((k / S) & 1));
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(C::TMEM_COLS) : "memory");
}

// ---------------------------------------------------------------------------
// weight and bias gradients of one layer on tcgen05
//
// Per tap, dW_tap = G^T A_tap is a contraction over pixels: K = 16 adjacent
// pixels of one row per MMA, both operands MN-major (a pixel's eight channels
// of one plane are 16 contiguous bytes, eight adjacent pixels one 128-byte core
// matrix), so tiles go from memory to the tensor cores without a transpose.
// TMA lands a tile as [row][plane][column][8 channels]: consecutive (row,
// plane) pairs are one plane row apart, so one operand can span several image
// rows with a single stride, and the taps' row offsets dy come out of one MMA:
//   GA = false (32 input channels): A operand = 4 activation rows x 32 channels
//     (M = 128), B operand = 2 gradient rows (N = 2 x 8 PG); block (ay, gy) of
//     the accumulator belongs to dy = ay - gy, 6 of the 8 blocks are taps;
//   GA = true (the first layer, one plane of inputs): A operand = 4 gradient
//     rows x 32 channels, B operand = 6 activation rows (N = 48).
// The column offset dx is a shifted start address: three accumulators. Per 32
// pixels of a 32-channel layer: 3 MMAs of 128 x 64 x 16, 6 KB of shared-memory
// reads each, 4.5 cycles per pixel and SM, under the 5.6 cycles that the
// 128 B/pixel take from HBM.
//
// One CTA per SM walks tiles of 16 x 32 pixels (18 x 34 activation halo; what
// lies outside the image reads as zero, so ragged tiles need no mask): lane 0
// of warp 0 requests tiles three stages ahead, lane 0 of warp 1 issues the
// MMAs, warps 2 and 3 sum the gradient tile for the bias. The accumulators
// stay in tensor memory until the CTA's last tile; each CTA then stores one
// partial gradient vector (layout [tap][cout][cin], then the bias), and
// wgrad_reduce_kernel adds the CTAs' vectors in a fixed order.
// 16 x 256^2, 32 x 32 channels: 34 us per launch (134 MB of activations and
// gradients, 4.0 TB/s); 180 us with mma.sync on tiles transposed through
// shared memory and one atomic per weight and CTA.
// ---------------------------------------------------------------------------
constexpr int kWgTW = 32, kWgTH = 16, kWgStages = 3;

template <bool GA, int PA, int PG>
struct WgradCfg {
    static constexpr int AW = kWgTW + 2, AR = kWgTH + 2;                  // activation tile with halo
    static constexpr int ABYTES = AR * PA * AW * 16, GBYTES = kWgTH * PG * kWgTW * 16;
    static constexpr int ASTRIDE = (ABYTES + 127) / 128 * 128;             // TMA destinations on 128 bytes
    static constexpr int STAGE = ASTRIDE + GBYTES;
    static constexpr int STEP = GA ? 4 : 2;                                // output rows per MMA
    static constexpr int N = GA ? 8 * PA * (STEP + 2) : 8 * PG * STEP;     // accumulator columns per dx
    static constexpr int TMEM_COLS = 3 * N <= 64 ? 64 : (3 * N <= 128 ? 128 : 256);
    static constexpr int COUT = 8 * PG;
    static_assert(GBYTES % 128 == 0 && N % 16 == 0 && 3 * N <= 256, "tile");
    static_assert(GA ? PG == 4 : PA == 4, "the A operand spans 128 rows");
    // epilogue scratch (reuses the stages): GA = false 9 COUT x 32 floats, GA =
    // true 4 x 18 x 32; the bias sums of two warps follow
    static constexpr int SCRATCH = (GA ? 4 * 9 * 2 * 32 : 9 * COUT * 32) * (int)sizeof(float);
    static_assert(SCRATCH <= kWgStages * STAGE, "scratch fits the stages");
    static constexpr size_t SMEM = (size_t)kWgStages * STAGE + 128;        // + alignment of the first stage
};

// instruction descriptor as idesc_m128, both operands MN-major
__host__ __device__ constexpr uint32_t idesc_m128_mn(uint32_t n) { return idesc_m128(n) | (1u << 15) | (1u << 16); }

// floats of one CTA's partial vector of a layer (real channels)
__host__ __device__ constexpr int wgrad_part(int cin, int cout) { return 9 * cin * cout + cout; }

// ta, tg: TMA views of the activations [img][PA][H][W][8] and gradients
// [img][PG][H][W][8] (see wgrad); part: gridDim.x partial vectors
template <bool GA, int PA, int PG>
__global__ void __launch_bounds__(128)
conv3x3_wgrad_tc(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tg,
                 float* __restrict__ part, int cin, int cout, int H, int W, int images, NetErr* __restrict__ err) {
    using C = WgradCfg<GA, PA, PG>;
    extern __shared__ unsigned char wg_raw[];
    __shared__ __align__(8) unsigned long long full[kWgStages], empty[kWgStages], done;
    __shared__ uint32_t tmem_base;
    __shared__ float sDb[2][32];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* sm = wg_raw + ((128u - (sh_addr(wg_raw) & 127u)) & 127u);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sh_addr(&tmem_base)),
                     "n"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kWgStages; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sh_addr(&full[i])) : "memory");
            // a stage is free once its MMAs and both bias warps are done with it
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 3;" ::"r"(sh_addr(&empty[i])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sh_addr(&done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    layer_release();
    layer_wait();
    const uint32_t tmem = tmem_base;
    const int tiles_x = (W + kWgTW - 1) / kWgTW, per_img = tiles_x * ((H + kWgTH - 1) / kWgTH);
    const int ntiles = per_img * images, G = gridDim.x;
    bool ok = true;
    int asked = 0;                                   // (producer) copies requested
    float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (warp == 0 && lane == 0) {
        int i = 0;
        for (int t = blockIdx.x; t < ntiles; t += G, ++i) {
            const int s = i % kWgStages;
            if (i >= kWgStages && !mbar_wait_bounded(sh_addr(&empty[s]), (uint32_t)((i / kWgStages - 1) & 1))) {
                ok = false;
                break;
            }
            const int img = t / per_img, rem = t - img * per_img;
            const int y0 = (rem / tiles_x) * kWgTH, x0 = (rem % tiles_x) * kWgTW;
            const uint32_t bar = sh_addr(&full[s]), dst = sh_addr(sm + s * C::STAGE);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(C::ABYTES + C::GBYTES)
                         : "memory");
            // x in 4-byte elements, four per pixel and plane: 16-byte aligned; pixels
            // outside the image read as zero
            asm volatile(
                "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
                "%5}], [%6];" ::"r"(dst),
                "l"(reinterpret_cast<uint64_t>(&ta)), "r"((x0 - 1) * 4), "r"(0), "r"(y0 - 1), "r"(img), "r"(bar)
                : "memory");
            asm volatile(
                "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
                "%5}], [%6];" ::"r"(dst + C::ASTRIDE),
                "l"(reinterpret_cast<uint64_t>(&tg)), "r"(x0 * 4), "r"(0), "r"(y0), "r"(img), "r"(bar)
                : "memory");
            asked = i + 1;
        }
        // every stage's last release has arrived before the CTA ends
        for (int k = i > kWgStages ? i - kWgStages : 0; ok && k < i; ++k)
            ok = mbar_wait_bounded(sh_addr(&empty[k % kWgStages]), (uint32_t)((k / kWgStages) & 1));
    } else if (warp == 1 && lane == 0) {
        int i = 0;
        for (int t = blockIdx.x; t < ntiles; t += G, ++i) {
            const int s = i % kWgStages;
            if (!mbar_wait_bounded(sh_addr(&full[s]), (uint32_t)((i / kWgStages) & 1))) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t aB = sh_addr(sm + s * C::STAGE), gB = aB + C::ASTRIDE;
#pragma unroll 1
            for (int r = 0; r < kWgTH; r += C::STEP) {
#pragma unroll
                for (int kc = 0; kc < kWgTW / 16; ++kc) {
                    const uint32_t gAddr = gB + (uint32_t)(r * PG * kWgTW + 16 * kc) * 16;
                    const uint64_t gd = umma_desc(gAddr, 128, kWgTW * 16);
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        const uint64_t ad = umma_desc(aB + (uint32_t)(r * PA * C::AW + 16 * kc + dx) * 16, 128,
                                                      C::AW * 16);
                        umma_f16(tmem + (uint32_t)(C::N * dx), GA ? gd : ad, GA ? ad : gd, idesc_m128_mn(C::N),
                                 (i | r | kc) != 0 ? 1u : 0u);
                    }
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             sh_addr(&empty[s]))
                         : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(sh_addr(&done))
                     : "memory");
    } else if (warp >= 2) {
        // bias: thread j of the 64 sums plane j % PG over every (64 / PG)-th pixel
        const int j = tid - 64, pl = j % PG;
        int i = 0;
        for (int t = blockIdx.x; t < ntiles; t += G, ++i) {
            const int s = i % kWgStages;
            // (one answer for the warp, as its lanes meet again below)
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(sh_addr(&full[s]), (uint32_t)((i / kWgStages) & 1)));
            if (!ok) break;
            const uint4* g4 = reinterpret_cast<const uint4*>(sm + s * C::STAGE + C::ASTRIDE);
#pragma unroll 4
            for (int px = j / PG; px < kWgTW * kWgTH; px += 64 / PG) {
                const uint4 v = g4[((px / kWgTW) * PG + pl) * kWgTW + px % kWgTW];
                const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    db[2 * h] += __uint_as_float(w[h] << 16);
                    db[2 * h + 1] += __uint_as_float(w[h] & 0xFFFF0000u);
                }
            }
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(sh_addr(&empty[s])) : "memory");
        }
    }
    __syncwarp();
    ok = __syncthreads_and(ok) != 0;
    // the accumulators are complete (and, on a failure, every MMA issued is:
    // the commit above tracks all of them)
    ok = __syncthreads_and(mbar_wait_bounded(sh_addr(&done), 0u) && ok) != 0;
    if (!ok) {
        // a wait ran out: let the copies still in flight land (bounded) before leaving
        if (tid == 0) {
            net_fail(err);
            for (int i = asked > kWgStages ? asked - kWgStages : 0; i < asked; ++i)
                mbar_wait_bounded(sh_addr(&full[i % kWgStages]), (uint32_t)((i / kWgStages) & 1));
        }
    } else {
        tc_fence_after();
        float* __restrict__ mine = part + (size_t)blockIdx.x * wgrad_part(cin, cout);
        float* scr = reinterpret_cast<float*>(sm);
        const uint32_t tw = tmem + ((uint32_t)(32 * warp) << 16);
        if (warp >= 2) {
            // lanes with the same plane add up: 32 / PG lanes per plane
#pragma unroll
            for (int e = 0; e < 8; ++e) {
#pragma unroll
                for (int o = 16; o >= PG; o >>= 1) db[e] += __shfl_down_sync(0xffffffffu, db[e], o);
                if (lane < PG) sDb[warp - 2][8 * lane + e] = db[e];
            }
        }
        if constexpr (!GA) {
            // lane = input channel, warp = activation row ay; columns: gradient row gy, output channel
            constexpr int CO = C::COUT;
            for (int gy = 0; gy < 2; ++gy) {
                const int dy = warp - gy;
                if (gy == 1) __syncthreads();        // the rows of gy = 0 are in the scratch
                if (dy < 0 || dy > 2) continue;
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                    for (int q = 0; q < CO; q += CO < 16 ? 8 : 16) {
                        constexpr int NV = CO < 16 ? 8 : 16;
                        float v[NV];
                        tmem_ld(tw + (uint32_t)(C::N * dx + CO * gy + q), v);
#pragma unroll
                        for (int c = 0; c < NV; ++c) {
                            const int tap = 3 * dy + dx;
                            float* sp = scr + (tap * CO + q + c) * 32 + lane;
                            if (gy == 0) *sp = v[c];
                            // (the rows of gy = 0 cover every dy, so each entry is complete here)
                            else if (q + c < cout) mine[(tap * cout + q + c) * 32 + lane] = *sp + v[c];
                        }
                    }
                }
            }
        } else {
            // lane = output channel, warp = gradient row gy; columns: activation row ay = gy + dy, input channel
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    float v[8];
                    tmem_ld(tw + (uint32_t)(C::N * dx + 8 * (warp + dy)), v);
                    scr[((warp * 9 + 3 * dy + dx) * 2 + 0) * 32 + lane] = v[0];
                    scr[((warp * 9 + 3 * dy + dx) * 2 + 1) * 32 + lane] = v[1];
                }
            }
            __syncthreads();
            for (int e = tid; e < 9 * 2 * 32; e += 128) {
                const int co = e & 31, ci = (e >> 5) & 1, tap = e >> 6;
                float v = 0.f;
#pragma unroll
                for (int gy = 0; gy < 4; ++gy) v += scr[((gy * 9 + tap) * 2 + ci) * 32 + co];
                mine[(tap * 32 + co) * 2 + ci] = v;
            }
        }
        __syncthreads();
        if (tid < cout) mine[9 * cin * cout + tid] = sDb[0][tid] + sDb[1][tid];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(C::TMEM_COLS) : "memory");
}

// The layers' gradients from the CTAs' partial vectors (ncta per layer, added
// in a fixed order). Block: 32 entries of one partial vector x 8 shares of the
// CTAs. ws: per layer ncta x wgrad_part floats, at ncta * base.
struct ReduceArgs {
    int cin[kLayers], cout[kLayers], block0[kLayers + 1];
    long long base[kLayers], param[kLayers];
};
__global__ void __launch_bounds__(256)
wgrad_reduce_kernel(const float* __restrict__ ws, float* __restrict__ grads, int ncta, ReduceArgs a) {
    __shared__ float red[8][33];
    int l = 0;
    while (l + 1 < kLayers && (int)blockIdx.x >= a.block0[l + 1]) ++l;
    const int cin = a.cin[l], cout = a.cout[l], n = wgrad_part(cin, cout);
    const int lane = threadIdx.x & 31, sh = threadIdx.x >> 5;
    const int e = ((int)blockIdx.x - a.block0[l]) * 32 + lane;
    float v = 0.f;
    if (e < n) {
        const float* p = ws + a.base[l] * ncta + e;
#pragma unroll 4
        for (int c = sh; c < ncta; c += 8) v += p[(size_t)c * n];
    }
    red[sh][lane] = v;
    __syncthreads();
    if (sh == 0 && e < n) {
        v = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) v += red[k][lane];
        const int nw = 9 * cin * cout;
        // partial [tap][cout][cin] -> parameters w[cout][cin][3][3], then the bias
        int o = e;
        if (e < nw) {
            const int tap = e / (cin * cout), co = (e / cin) % cout, ci = e % cin;
            o = (co * cin + ci) * 9 + tap;
        }
        grads[a.param[l] + o] = v;
    }
}

// ---------------------------------------------------------------------------
// loss and its gradient in the output: g = 2 c_k (o - t) / npx (one plane of
// eight channels, 4 used; its readers take the second plane of a 16-channel
// operand as zeros outside the tensor map). 48 B per pixel and four FMAs on the
// few FP64 units, where a squared error is exact (48 bits, any finite float's
// square in range) and so are infinities and NaN. Normal floats are widened with
// integer instructions, since conversions run on those units as well. One atomic
// per block; the grid is a few blocks per SM, not one block per 256 pixels: 4096
// atomics on one address and eight FP64 operations per pixel made it 50 us at
// 16 x 256^2, now 18 us (26 with conversions).
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool is_normal(float v) {
    return (__float_as_uint(v) & 0x7FFFFFFFu) - 0x00800000u < 0x7F000000u;
}
// |v| of a normal float: the exponent moved by 1023 - 127, the fraction by 29 bits
__device__ __forceinline__ double widen_abs(float v) {
    const uint32_t u = __float_as_uint(v) & 0x7FFFFFFFu;
    return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}

__global__ void __launch_bounds__(256)
cnn_loss_kernel(const float* __restrict__ o, const float* __restrict__ tg, float4 cw, bf16* __restrict__ gout,
                double* __restrict__ loss, long long npx) {
    __shared__ double red[8];
    double sx = 0.0, sy = 0.0, sz = 0.0, sw = 0.0;   // sums of the squared errors
    const float s = 2.0f / (float)npx;
    for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < npx; i += (long long)gridDim.x * 256) {
        const float4 ov = reinterpret_cast<const float4*>(o)[i];
        const float4 tv = __ldcs(reinterpret_cast<const float4*>(tg) + i);
        const float e0 = ov.x - tv.x, e1 = ov.y - tv.y, e2 = ov.z - tv.z, e3 = ov.w - tv.w;
        double d0, d1, d2, d3;
        if (is_normal(e0) && is_normal(e1) && is_normal(e2) && is_normal(e3)) {
            d0 = widen_abs(e0);
            d1 = widen_abs(e1);
            d2 = widen_abs(e2);
            d3 = widen_abs(e3);
        } else {
            d0 = e0;
            d1 = e1;
            d2 = e2;
            d3 = e3;
        }
        sx = fma(d0, d0, sx);
        sy = fma(d1, d1, sy);
        sz = fma(d2, d2, sz);
        sw = fma(d3, d3, sw);
        reinterpret_cast<uint4*>(gout)[i] =
            make_uint4(pack2(__float2bfloat16(s * cw.x * e0), __float2bfloat16(s * cw.y * e1)),
                       pack2(__float2bfloat16(s * cw.z * e2), __float2bfloat16(s * cw.w * e3)), 0u, 0u);
    }
    double l = (double)cw.x * sx + (double)cw.y * sy + (double)cw.z * sz + (double)cw.w * sw;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l += __shfl_down_sync(0xffffffffu, l, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        atomicAdd(loss, t / (double)npx);
    }
}

// ---------------------------------------------------------------------------
// Adam (Kingma and Ba, Algorithm 1) on the FP32 parameter vector
// ---------------------------------------------------------------------------
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ gd, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps,
                            float c1, float c2, NetErr* __restrict__ err) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (err->flag) {                     // the gradients are not whole: no step
        if (i == 0) ++err->skipped;
        return;
    }
    const float gi = gd[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---------------------------------------------------------------------------
// BF16 weight packing: forward [tap][coutp][cinp], and for the input
// gradient the flipped transpose [tap'][cinp][coutp_g] with
// w'[tap'][i][o] = w[o][i][8 - tap'] (zero in the padding)
// ---------------------------------------------------------------------------
__global__ void pack_kernel(const float* __restrict__ w, bf16* __restrict__ fwd, bf16* __restrict__ bwd,
                            int cin, int cout, int cinp, int coutp, int coutg) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int nf = 9 * coutp * cinp;
    if (e < nf) {
        const int tap = e / (coutp * cinp), o = (e / cinp) % coutp, i = e % cinp;
        const float x = (o < cout && i < cin) ? w[((size_t)o * cin + i) * 9 + tap] : 0.f;
        fwd[e] = __float2bfloat16(x);
    }
    const int nb = 9 * cinp * coutg;
    if (bwd && e < nb) {
        const int tap = e / (cinp * coutg), i = (e / coutg) % cinp, o = e % coutg;
        const float x = (o < cout && i < cin) ? w[((size_t)o * cin + i) * 9 + (8 - tap)] : 0.f;
        bwd[e] = __float2bfloat16(x);
    }
}

// ---------------------------------------------------------------------------
// output -> warm start (x0, d1, (d2h, d2v) interleaved)
// ---------------------------------------------------------------------------
__global__ void split_start_kernel(const float* __restrict__ o, float s0, float s1, float s2,
                                   float* __restrict__ x0, float* __restrict__ d0, long long n, long long npx) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npx) return;
    const long long im = i / n, px = i % n;
    const float4 v = reinterpret_cast<const float4*>(o)[i];
    x0[i] = s0 * v.x;
    float* d = d0 + im * 3 * n;
    d[px] = s1 * v.y;
    reinterpret_cast<float2*>(d + n)[px] = make_float2(s2 * v.z, s2 * v.w);
}

// the same two steps for a group of separately stored problems (the learned
// start of a batch solve): per-image device pointers, passed by value
struct ImgPtrs {
    const float* y[kWsBatch];
    const uint8_t* m[kWsBatch];
    float* x0[kWsBatch];
    float* d0[kWsBatch];
};

// grid (ceil(hw / 256), images)
__global__ void cnn_input_ptrs_kernel(ImgPtrs P, bf16* __restrict__ a0, long long hw) {
    const long long px = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (px >= hw) return;
    const int img = blockIdx.y;
    const bool obs = P.m[img][px] != 0;
    const float y = obs ? P.y[img][px] : 0.f;
    reinterpret_cast<uint4*>(a0)[(long long)img * hw + px] =
        make_uint4(pack2(__float2bfloat16(y), __float2bfloat16(obs ? 1.f : 0.f)), 0u, 0u, 0u);
}

// grid (ceil(hw / 256), images)
__global__ void split_start_ptrs_kernel(const float* __restrict__ o, float s0, float s1, float s2, ImgPtrs P,
                                        long long hw) {
    const long long px = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (px >= hw) return;
    const int img = blockIdx.y;
    const float4 v = reinterpret_cast<const float4*>(o)[(long long)img * hw + px];
    P.x0[img][px] = s0 * v.x;
    float* d = P.d0[img];
    d[px] = s1 * v.y;
    reinterpret_cast<float2*>(d + hw)[px] = make_float2(s2 * v.z, s2 * v.w);
}

// ---------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------
// the driver's tensor-map encoder (through the runtime, no link to the driver library)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// launch a layer of the chain; first: as a plain launch
template <typename... KArgs, typename... Args>
cudaError_t launch_layer(void (*kern)(KArgs...), bool first, int grid, int block, size_t smem, cudaStream_t s,
                         Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = first ? 0 : 1;
    ++g_cnn_launches;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// One layer on tcgen05 (persistent CTAs over 8 x 16 tiles, as many per SM as
// registers, shared memory and tensor memory allow). The input planes [img][CIN / 8][H][W][8] are viewed by TMA as a 4-D tensor
// (8 W elements of a plane row, H, CIN / 8 planes, images) with strides
// (16 W, 16 W H, 16 W H CIN / 8) bytes, and a box of (80, 18, CIN / 8, 1):
// one halo tile per copy, laid out in shared memory as
// [plane][halo row][halo column][8 channels].
template <int CIN, int MODE>
cudaError_t conv_tc(bool first, const bf16* in, const bf16* w, const float* bias, void* out, const bf16* gate,
                    int count, int H, int W, int sms, NetErr* err, cudaStream_t s) {
    static int per_sm = 0;
    if (per_sm == 0) {
        // CTAs one SM holds, from the kernel's registers and static shared
        // memory (the whole unified L1 / shared array given to shared memory)
        // and the 2 x cout tensor-memory columns each CTA allocates of 512
        cudaFuncAttributes fa;
        int dev = 0, smem_sm = 0, smem_rsv = 0, regs_sm = 0;
        if (cudaFuncSetAttribute(conv3x3_tc<CIN, MODE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, conv3x3_tc<CIN, MODE>) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&smem_rsv, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess)
            return cudaErrorInvalidConfiguration;
        const int regs_cta = ((fa.numRegs + 7) / 8) * 8 * 128;
        const int by_regs = regs_sm / std::max(regs_cta, 1);
        const int by_smem = smem_sm / (int)(fa.sharedSizeBytes + smem_rsv);
        const int cout = MODE == kModeOutF32 ? 16 : 32;
        per_sm = std::max(1, std::min({by_regs, by_smem, 16, 512 / (2 * cout)}));
    }
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap tm;
    const cuuint64_t plane = (cuuint64_t)W * H * 16;
    constexpr int PL = stored_planes(CIN);       // (a plane outside the map reads as zero)
    const cuuint64_t dims[4] = {(cuuint64_t)W * 8, (cuuint64_t)H, (cuuint64_t)PL, (cuuint64_t)count};
    const cuuint64_t strides[3] = {(cuuint64_t)W * 16, plane, plane * PL};
    const cuuint32_t box[4] = {(cuuint32_t)kTcHW * 8, (cuuint32_t)kTcHH, (cuuint32_t)(CIN / 8), 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    if (enc(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(in), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    const int ntiles = (W / kTcTW) * (H / kTcTH) * count;
    const int grid = std::min(ntiles, per_sm * sms);
    return launch_layer(conv3x3_tc<CIN, MODE>, first, grid, 128, 0, s, tm, w, bias, out, gate, H, W, count, err);
}

// Strips of 128 columns against 8 x 16 tiles: a strip costs the same however
// much of it lies in the image, and the tiles take 1.23 times the strips' time
// on full strips (103 / 126 us per hidden layer at 16 x 512^2), so the strips
// are taken while they are at most a quarter wider than the image.
bool rows_fit(int W) { return ((W + kStrip - 1) / kStrip) * kStrip * 4 <= W * 5; }

// One layer of 16 or 32 input channels: conv3x3_rows where its strips of 128
// columns fit the width, else the 8 x 16 tiles of conv3x3_tc
template <int CIN, int MODE>
cudaError_t conv_rows(const bf16* in, const bf16* w, const float* bias, void* out, const bf16* gate, int count,
                      int H, int W, int sms, NetErr* err, cudaStream_t s, const StartOut& st = StartOut{}) {
    using C = RowsCfg<CIN, MODE>;
    const int strips = (W + kStrip - 1) / kStrip;
    if constexpr (MODE != kModeStart) {
        if (!rows_fit(W)) return conv_tc<CIN, MODE>(false, in, w, bias, out, gate, count, H, W, sms, err, s);
    }
    cudaError_t e = cudaFuncSetAttribute(conv3x3_rows<CIN, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)C::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(conv3x3_rows<CIN, MODE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    // (at least eight strip rows per CTA: each segment adds two halo rows)
    const long long total = (long long)count * strips * H;
    const int grid = (int)std::max(1LL, std::min((long long)C::CTAS * sms, total / 8));
    return launch_layer(conv3x3_rows<CIN, MODE>, false, grid, 192, C::SMEM, s, in, w, bias, out, gate, H, W, count, err,
                        st);
}

// One layer's weight and bias gradients into the CTAs' partial vectors. The
// planes are viewed by TMA as 4-D tensors (4 W four-byte elements of a plane
// row, planes, H, images), so that a tile lands as [row][plane][column][8].
template <bool GA, int PA, int PG>
cudaError_t wgrad(bool first, const bf16* a, const bf16* g, float* part, int cin, int cout, int count, int H, int W,
                  int grid, NetErr* err, cudaStream_t s) {
    using C = WgradCfg<GA, PA, PG>;
    cudaError_t e = cudaFuncSetAttribute(conv3x3_wgrad_tc<GA, PA, PG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)C::SMEM);
    if (e != cudaSuccess) return e;
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc) return cudaErrorNotSupported;
    CUtensorMap tm[2];
    for (int k = 0; k < 2; ++k) {
        const cuuint64_t np = k == 0 ? PA : PG, plane = (cuuint64_t)W * H * 16;
        const cuuint64_t dims[4] = {(cuuint64_t)W * 4, np, (cuuint64_t)H, (cuuint64_t)count};
        const cuuint64_t strides[3] = {plane, (cuuint64_t)W * 16, plane * np};
        const cuuint32_t box[4] = {(cuuint32_t)(k == 0 ? C::AW : kWgTW) * 4, (cuuint32_t)np,
                                   (cuuint32_t)(k == 0 ? C::AR : kWgTH), 1};
        const cuuint32_t es[4] = {1, 1, 1, 1};
        if (enc(&tm[k], CU_TENSOR_MAP_DATA_TYPE_UINT32, 4, const_cast<bf16*>(k == 0 ? a : g), dims, strides, box, es,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    return launch_layer(conv3x3_wgrad_tc<GA, PA, PG>, first, grid, 128, C::SMEM, s, tm[0], tm[1], part, cin, cout, H, W,
                        count, err);
}

}  // namespace

struct admm_cnn_s {
    int device = 0;
    int sms = 152;
    long long max_px = 0;
    bool training = false;
    float* params = nullptr;       // FP32 master vector
    float* grads = nullptr;
    float* m = nullptr;
    float* v = nullptr;
    long long adam_t = 0;
    bf16* wf[kLayers] = {};        // packed forward weights
    bf16* wb[kLayers] = {};        // packed input-gradient weights (layers 1..)
    bf16* a0 = nullptr;            // input, one plane of 8 channels
    bf16* act[kLayers - 1] = {};   // activations after layers 0..6 (training keeps all)
    float* out = nullptr;          // output, 4 channels FP32
    bf16* gbuf[2] = {};            // gradient ping-pong, 32 channels
    bf16* gout = nullptr;          // output gradient, one plane of 8 channels
    float* wpart = nullptr;        // weight-gradient partial vectors, one per CTA and layer
    double* loss = nullptr;        // device accumulator
    double* h_loss = nullptr;      // pinned
    NetErr* err = nullptr;         // set by a convolution whose bounded wait ran out
    int* h_err = nullptr;          // ... and its pinned flag
    std::vector<void*> allocs;
};

namespace {

template <typename T>
int dalloc(admm_cnn_s* n, T** p, size_t count) {
    void* q = nullptr;
    if (admm::alloc_fault_fire()) return ADMM_ENOMEM;
    if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        return ADMM_ENOMEM;
    }
    n->allocs.push_back(q);
    *p = static_cast<T*>(q);
    return ADMM_OK;
}

int check_shape(const admm_cnn_s* n, int count, int H, int W) {
    if (count <= 0 || H < kTile || W < kTile || H % kTile || W % kTile) return ADMM_EINVAL;
    if ((long long)count * H * W > n->max_px) return ADMM_EINVAL;
    return ADMM_OK;
}

// a kernel of an earlier call, or of this one once it has been waited for, ran
// into its limit
bool net_failed(const admm_cnn_s* n) { return *static_cast<volatile const int*>(n->h_err) != 0; }
// the code for it, once: waits for the device, takes the steps that were left
// out off Adam's count and clears the state
int net_report(admm_cnn_s* n) {
    NetErr e{};
    CKC(cudaDeviceSynchronize());
    CKC(cudaMemcpy(&e, n->err, sizeof(e), cudaMemcpyDeviceToHost));
    n->adam_t -= e.skipped;
    CKC(cudaMemset(n->err, 0, offsetof(NetErr, host)));
    CKC(cudaDeviceSynchronize());
    *static_cast<volatile int*>(n->h_err) = 0;
    return ADMM_ETIMEOUT;
}

int pack_all(admm_cnn_s* n, cudaStream_t s) {
    for (int l = 0; l < kLayers; ++l) {
        const int cin = layer_cin(l), cout = layer_cout(l);
        const int cinp = layer_cinp(l), coutp = layer_coutp(l);
        const int coutg = pad16(cout);
        const int nmax = std::max(9 * coutp * cinp, 9 * cinp * coutg);
        pack_kernel<<<(nmax + 255) / 256, 256, 0, s>>>(n->params + param_offset(l), n->wf[l], n->wb[l], cin, cout,
                                                        cinp, coutp, coutg);
        ++g_cnn_launches;
        CKC(cudaGetLastError());
    }
    return ADMM_OK;
}

// the eight layers on the prepared input n->a0; with `keep` every activation
// is stored for the backward pass, otherwise two buffers alternate. The output
// goes to `out` (16-byte aligned) or, with `st` (rows_fit(W) only), to a
// predicted start.
int run_layers(admm_cnn_s* n, int count, int H, int W, bool keep, float* out, const StartOut* st, cudaStream_t s) {
    const bf16* cur = n->a0;
    StartOut stall{};                    // (the test hook serves one pass)
    stall.test_stall = g_cnn_test_stall;
    g_cnn_test_stall = 0;
    for (int l = 0; l < kLayers; ++l) {
        const float* b = n->params + param_offset(l) + (long long)layer_cout(l) * layer_cin(l) * 9;
        if (l == kLayers - 1) {
            if (st)
                CKC((conv_rows<32, kModeStart>(cur, n->wf[l], b, nullptr, nullptr, count, H, W, n->sms, n->err, s,
                                               *st)));
            else
                CKC((conv_rows<32, kModeOutF32>(cur, n->wf[l], b, out, nullptr, count, H, W, n->sms, n->err, s)));
        } else {
            bf16* dst = keep ? n->act[l] : n->act[l & 1];
            if (l == 0)
                CKC((conv_tc<8, kModeReluBf16>(true, cur, n->wf[l], b, dst, nullptr, count, H, W, n->sms, n->err, s)));
            else
                CKC((conv_rows<32, kModeReluBf16>(cur, n->wf[l], b, dst, nullptr, count, H, W, n->sms, n->err, s,
                                                  l == 1 ? stall : StartOut{})));
            cur = dst;
        }
    }
    return ADMM_OK;
}

// forward pass from [M^T y, mask] stored contiguously for the count images
int forward(admm_cnn_s* n, int count, int H, int W, const float* ybar, const uint8_t* mask, bool keep, float* out,
            const StartOut* st, cudaStream_t s) {
    const long long npx = (long long)count * H * W;
    cnn_input_kernel<<<(unsigned)((npx + 255) / 256), 256, 0, s>>>(ybar, mask, n->a0, npx);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    return run_layers(n, count, H, W, keep, out, st, s);
}

// loss, gradients into n->grads
int backward(admm_cnn_s* n, int count, int H, int W, const float* target, const float* chan_w, cudaStream_t s) {
    const long long npx = (long long)count * H * W;
    CKC(cudaMemsetAsync(n->loss, 0, sizeof(double), s));
    const float4 cw = make_float4(chan_w[0], chan_w[1], chan_w[2], chan_w[3]);
    const unsigned lgrid = (unsigned)std::min((npx + 255) / 256, 6LL * n->sms);
    cnn_loss_kernel<<<lgrid, 256, 0, s>>>(n->out, target, cw, n->gout, n->loss, npx);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    const int tiles = ((H + kWgTH - 1) / kWgTH) * ((W + kWgTW - 1) / kWgTW) * count;
    const int ncta = std::min(tiles, n->sms);
    ReduceArgs ra{};
    long long base = 0;
    int blocks = 0;
    for (int l = 0; l < kLayers; ++l) {
        const int np = wgrad_part(layer_cin(l), layer_cout(l));
        ra.cin[l] = layer_cin(l);
        ra.cout[l] = layer_cout(l);
        ra.base[l] = base;
        ra.param[l] = param_offset(l);
        ra.block0[l] = blocks;
        base += np;
        blocks += (np + 31) / 32;
    }
    ra.block0[kLayers] = blocks;
    const bf16* g = n->gout;                        // gradient in the output of layer l
    for (int l = kLayers - 1; l >= 0; --l) {
        float* pt = n->wpart + ra.base[l] * ncta;
        const bf16* a_in = l == 0 ? n->a0 : n->act[l - 1];
        if (l == kLayers - 1)
            CKC((wgrad<false, 4, 1>(true, a_in, g, pt, kWidth, kOut, count, H, W, ncta, n->err, s)));
        else if (l == 0)
            CKC((wgrad<true, 1, 4>(false, a_in, g, pt, kIn, kWidth, count, H, W, ncta, n->err, s)));
        else
            CKC((wgrad<false, 4, 4>(false, a_in, g, pt, kWidth, kWidth, count, H, W, ncta, n->err, s)));
        if (l == 0) break;
        bf16* gnext = n->gbuf[l & 1];
        if (l == kLayers - 1)
            CKC((conv_rows<16, kModeGateBf16>(g, n->wb[l], nullptr, gnext, a_in, count, H, W, n->sms, n->err, s)));
        else
            CKC((conv_rows<32, kModeGateBf16>(g, n->wb[l], nullptr, gnext, a_in, count, H, W, n->sms, n->err, s)));
        g = gnext;
    }
    wgrad_reduce_kernel<<<blocks, 256, 0, s>>>(n->wpart, n->grads, ncta, ra);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    return ADMM_OK;
}

}  // namespace

extern "C" {

long long admm_cnn_param_count(void) { return param_count(); }

long long admm_cnn_launches(void) {
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    return g_cnn_launches;
}

void admm_cnn_destroy(admm_cnn_t net) {
    if (!net) return;
    for (void* p : net->allocs) cudaFree(p);
    if (net->h_loss) cudaFreeHost(net->h_loss);
    if (net->h_err) cudaFreeHost(net->h_err);
    delete net;
}

int admm_cnn_create(admm_cnn_t* out, long long max_pixels, int training) {
    if (!out || max_pixels <= 0) return ADMM_EINVAL;
    *out = nullptr;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    admm_cnn_s* n = new (std::nothrow) admm_cnn_s();
    if (!n) return ADMM_ENOMEM;
    int rc = ADMM_OK;
    auto bail = [&](int r) {
        admm_cnn_destroy(n);
        return r;
    };
    if (cudaGetDevice(&n->device) != cudaSuccess) return bail(ADMM_ECUDA);
    cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, n->device);
    n->max_px = max_pixels;
    n->training = training != 0;
    const long long P = param_count();
    const size_t px = (size_t)max_pixels;
    if ((rc = dalloc(n, &n->params, P)) || (rc = dalloc(n, &n->a0, px * 8)) || (rc = dalloc(n, &n->out, px * 4)) ||
        (rc = dalloc(n, &n->err, 1)))
        return bail(rc);
    for (int l = 0; l < kLayers; ++l) {
        if ((rc = dalloc(n, &n->wf[l], (size_t)9 * layer_coutp(l) * layer_cinp(l)))) return bail(rc);
        if (l > 0 && (rc = dalloc(n, &n->wb[l], (size_t)9 * layer_cinp(l) * pad16(layer_cout(l))))) return bail(rc);
    }
    const int nact = n->training ? kLayers - 1 : 2;
    for (int l = 0; l < nact; ++l)
        if ((rc = dalloc(n, &n->act[l], px * kWidth))) return bail(rc);
    if (n->training) {
        if ((rc = dalloc(n, &n->grads, P)) || (rc = dalloc(n, &n->m, P)) || (rc = dalloc(n, &n->v, P)) ||
            (rc = dalloc(n, &n->gbuf[0], px * kWidth)) || (rc = dalloc(n, &n->gbuf[1], px * kWidth)) ||
            (rc = dalloc(n, &n->gout, px * 8)) || (rc = dalloc(n, &n->loss, 1)) ||
            (rc = dalloc(n, &n->wpart, (size_t)P * n->sms)))
            return bail(rc);
        if (admm::alloc_fault_fire() || cudaHostAlloc(&n->h_loss, sizeof(double), cudaHostAllocDefault) != cudaSuccess) {
            n->h_loss = nullptr;
            return bail(ADMM_ENOMEM);
        }
    }
    if (cudaMemset(n->params, 0, P * sizeof(float)) != cudaSuccess) return bail(ADMM_ECUDA);
    if (admm::alloc_fault_fire() || cudaHostAlloc(&n->h_err, sizeof(int), cudaHostAllocMapped) != cudaSuccess) {
        n->h_err = nullptr;
        cudaGetLastError();
        return bail(ADMM_ENOMEM);
    }
    *n->h_err = 0;
    NetErr e{};
    if (cudaHostGetDevicePointer(&e.host, n->h_err, 0) != cudaSuccess ||
        cudaMemcpy(n->err, &e, sizeof(e), cudaMemcpyHostToDevice) != cudaSuccess)
        return bail(ADMM_ECUDA);
    if (pack_all(n, nullptr) != ADMM_OK || cudaDeviceSynchronize() != cudaSuccess) return bail(ADMM_ECUDA);
    *out = n;
    return ADMM_OK;
}

int admm_cnn_set_params(admm_cnn_t net, const float* params) {
    if (!net || !params) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    if (net_failed(net)) return net_report(net);
    const long long P = param_count();
    CKC(cudaMemcpy(net->params, params, P * sizeof(float), cudaMemcpyDefault));
    if (net->training) {
        CKC(cudaMemset(net->m, 0, P * sizeof(float)));
        CKC(cudaMemset(net->v, 0, P * sizeof(float)));
        net->adam_t = 0;
    }
    const int rc = pack_all(net, nullptr);
    if (rc != ADMM_OK) return rc;
    CKC(cudaDeviceSynchronize());
    return ADMM_OK;
}

int admm_cnn_get_params(admm_cnn_t net, float* params) {
    if (!net || !params) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    CKC(cudaMemcpy(params, net->params, param_count() * sizeof(float), cudaMemcpyDefault));
    return net_failed(net) ? net_report(net) : ADMM_OK;
}

int admm_cnn_forward(admm_cnn_t net, int count, int H, int W, const float* ybar, const uint8_t* mask, float* out,
                     void* stream) {
    if (!net || !ybar || !mask || !out) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    int rc = check_shape(net, count, H, W);
    if (rc != ADMM_OK) return rc;
    if (net_failed(net)) return net_report(net);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // (the last layer stores 16 bytes per pixel: straight to `out` where that is aligned)
    const bool direct = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
    if ((rc = forward(net, count, H, W, ybar, mask, false, direct ? out : net->out, nullptr, s)) != ADMM_OK) return rc;
    if (!direct)
        CKC(cudaMemcpyAsync(out, net->out, (size_t)count * H * W * 4 * sizeof(float), cudaMemcpyDeviceToDevice, s));
    return ADMM_OK;
}

int admm_cnn_gradients(admm_cnn_t net, int count, int H, int W, const float* ybar, const uint8_t* mask,
                       const float* target, const float* chan_w, float* grads, double* loss, void* stream) {
    if (!net || !ybar || !mask || !target || !chan_w || !grads || !net->training) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    int rc = check_shape(net, count, H, W);
    if (rc != ADMM_OK) return rc;
    if (net_failed(net)) return net_report(net);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if ((rc = forward(net, count, H, W, ybar, mask, true, net->out, nullptr, s)) != ADMM_OK) return rc;
    if ((rc = backward(net, count, H, W, target, chan_w, s)) != ADMM_OK) return rc;
    CKC(cudaMemcpyAsync(grads, net->grads, param_count() * sizeof(float), cudaMemcpyDefault, s));
    CKC(cudaMemcpyAsync(net->h_loss, net->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
    CKC(cudaStreamSynchronize(s));
    if (net_failed(net)) return net_report(net);
    if (loss) *loss = *net->h_loss;
    return ADMM_OK;
}

int admm_cnn_train_step(admm_cnn_t net, int count, int H, int W, const float* ybar, const uint8_t* mask,
                        const float* target, const float* chan_w, float lr, double* loss, void* stream) {
    if (!net || !ybar || !mask || !target || !chan_w || !net->training || !(lr > 0.f)) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    int rc = check_shape(net, count, H, W);
    if (rc != ADMM_OK) return rc;
    if (net_failed(net)) return net_report(net);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if ((rc = forward(net, count, H, W, ybar, mask, true, net->out, nullptr, s)) != ADMM_OK) return rc;
    if ((rc = backward(net, count, H, W, target, chan_w, s)) != ADMM_OK) return rc;
    net->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)net->adam_t));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)net->adam_t));
    const long long P = param_count();
    adam_kernel<<<(unsigned)((P + 255) / 256), 256, 0, s>>>(net->params, net->grads, net->m, net->v, P, lr, b1, b2,
                                                            1e-8f, c1, c2, net->err);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    if ((rc = pack_all(net, s)) != ADMM_OK) return rc;
    if (loss) {
        CKC(cudaMemcpyAsync(net->h_loss, net->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
        CKC(cudaStreamSynchronize(s));
        if (net_failed(net)) return net_report(net);
        *loss = *net->h_loss;
    }
    return ADMM_OK;
}

int admm_cnn_predict_start(admm_cnn_t net, int count, int H, int W, const float* ybar, const uint8_t* mask,
                           const float* scales, float* x0, float* d0, void* stream) {
    if (!net || !ybar || !mask || !scales || !x0 || !d0) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    int rc = check_shape(net, count, H, W);
    if (rc != ADMM_OK) return rc;
    if (net_failed(net)) return net_report(net);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    StartOut st{};
    st.s0 = scales[0];
    st.s1 = scales[1];
    st.s2 = scales[2];
    st.x0 = x0;
    st.d0 = d0;
    const bool fit = rows_fit(W);
    if ((rc = forward(net, count, H, W, ybar, mask, false, net->out, fit ? &st : nullptr, s)) != ADMM_OK) return rc;
    if (fit) return ADMM_OK;         // the last layer has written the start
    const long long n = (long long)H * W, npx = n * count;
    split_start_kernel<<<(unsigned)((npx + 255) / 256), 256, 0, s>>>(net->out, scales[0], scales[1], scales[2], x0,
                                                                     d0, n, npx);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    return ADMM_OK;
}

// ---------------------------------------------------------------------------
// The library-global warm-start network of admm_warmstart_load, used by
// admm_deconv_solve_batch(..., use_warmstart = 1, ...): parameters and scales
// on the host; the inference network is created on first use on the current
// device and grown to the largest image it meets.
// ---------------------------------------------------------------------------
namespace {
struct WarmStartNet {
    bool loaded = false;
    std::vector<float> params;
    float scales[4] = {0.f, 0.f, 0.f, 0.f};
    admm_cnn_t net = nullptr;
    int device = -1;
    long long cap = 0;
};
std::mutex g_ws_mutex;
WarmStartNet g_ws;
}  // namespace

int admm_warmstart_load(const char* path) {
    std::lock_guard<std::mutex> lk(g_ws_mutex);
    if (!path) {
        if (g_ws.net) admm_cnn_destroy(g_ws.net);
        g_ws = WarmStartNet();
        return ADMM_OK;
    }
    FILE* f = std::fopen(path, "rb");
    if (!f) return ADMM_EINVAL;
    char magic[8];
    int32_t version = 0, reserved = 0;
    int64_t count = 0;
    float scales[4];
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "ADMMCNN1", 8) == 0 &&
              std::fread(&version, sizeof(version), 1, f) == 1 && version == 1 &&
              std::fread(&reserved, sizeof(reserved), 1, f) == 1 &&
              std::fread(&count, sizeof(count), 1, f) == 1 && count == param_count() &&
              std::fread(scales, sizeof(float), 4, f) == 4;
    std::vector<float> params;
    if (ok) {
        params.resize((size_t)count);
        ok = std::fread(params.data(), sizeof(float), params.size(), f) == params.size();
        char extra;
        ok = ok && std::fread(&extra, 1, 1, f) == 0;   // nothing after the parameters
    }
    std::fclose(f);
    if (!ok) return ADMM_EINVAL;
    for (float v : params)
        if (!std::isfinite(v)) return ADMM_EINVAL;
    if (g_ws.net) admm_cnn_destroy(g_ws.net);
    g_ws = WarmStartNet();
    g_ws.params.swap(params);
    std::memcpy(g_ws.scales, scales, sizeof(scales));
    g_ws.loaded = true;
    return ADMM_OK;
}

}  // extern "C"

namespace admm {
// the driver's tensor-map encoder, for the other translation units (null when
// the driver does not provide it)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encode_fn() { return tensor_map_encoder(); }

void cnn_test_stall(int value) {
    std::lock_guard<std::mutex> lk(g_cnn_mutex);
    g_cnn_test_stall = value;
}

bool ws_loaded() {
    std::lock_guard<std::mutex> lk(g_ws_mutex);
    return g_ws.loaded;
}

// whether a pass of the network since the last call of this function ran into
// the limit of a bounded wait (its stream has been waited for): ADMM_ETIMEOUT,
// and the state is clear again
int ws_take_error() {
    std::lock_guard<std::mutex> lk(g_ws_mutex);
    std::lock_guard<std::mutex> lk2(g_cnn_mutex);
    return g_ws.net && net_failed(g_ws.net) ? net_report(g_ws.net) : ADMM_OK;
}

// images of H x W that one ws_predict_starts call takes: up to 16, and no
// more than 16 x 512 x 512 pixels (the network's buffers hold about 180 B per
// pixel)
int ws_batch_limit(int H, int W) {
    const long long px = std::max(1LL, (long long)H * W);
    return (int)std::max(1LL, std::min((long long)kWsBatch, 16LL * 512 * 512 / px));
}

// predicted starts of `count` H x W TV problems (count <= ws_batch_limit):
// for image i, [M^T y, mask] from ybar[i], mask[i], and x0[i] (H W floats)
// and d0[i] (3 H W floats in the layout of admm_deconv_get_state) written,
// device pointers, on `s`. One pass of the network over the group; each
// image's result has the bits of a pass over that image alone.
int ws_predict_starts(int count, int H, int W, const float* const* ybar, const uint8_t* const* mask,
                      float* const* x0, float* const* d0, cudaStream_t s) {
    if (count < 1 || count > ws_batch_limit(H, W)) return ADMM_EINVAL;
    std::lock_guard<std::mutex> lk(g_ws_mutex);
    if (!g_ws.loaded) return ADMM_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return ADMM_ECUDA;
    const long long hw = (long long)H * W, px = hw * count;
    if (!g_ws.net || g_ws.device != dev || g_ws.cap < px) {
        if (g_ws.net) {
            // (its passes of this call are not waited for yet)
            CKC(cudaDeviceSynchronize());
            const bool failed = net_failed(g_ws.net);
            admm_cnn_destroy(g_ws.net);
            g_ws.net = nullptr;
            if (failed) return ADMM_ETIMEOUT;
        }
        const long long cap = std::max(px, 512LL * 512LL);
        admm_cnn_t n = nullptr;
        int rc = admm_cnn_create(&n, cap, 0);
        if (rc != ADMM_OK) return rc;
        rc = admm_cnn_set_params(n, g_ws.params.data());
        if (rc != ADMM_OK) {
            admm_cnn_destroy(n);
            return rc;
        }
        g_ws.net = n;
        g_ws.device = dev;
        g_ws.cap = cap;
    }
    admm_cnn_s* net = g_ws.net;
    std::lock_guard<std::mutex> lk2(g_cnn_mutex);
    int rc = check_shape(net, count, H, W);
    if (rc != ADMM_OK) return rc;
    ImgPtrs P{};
    for (int i = 0; i < count; ++i) {
        if (!ybar[i] || !mask[i] || !x0[i] || !d0[i]) return ADMM_EINVAL;
        P.y[i] = ybar[i];
        P.m[i] = mask[i];
        P.x0[i] = x0[i];
        P.d0[i] = d0[i];
    }
    const dim3 grid((unsigned)((hw + 255) / 256), (unsigned)count);
    cnn_input_ptrs_kernel<<<grid, 256, 0, s>>>(P, net->a0, hw);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    StartOut st{};
    st.s0 = g_ws.scales[0];
    st.s1 = g_ws.scales[1];
    st.s2 = g_ws.scales[2];
    st.separate = 1;
    for (int i = 0; i < count; ++i) {
        st.px0[i] = x0[i];
        st.pd0[i] = d0[i];
    }
    const bool fit = rows_fit(W);
    if ((rc = run_layers(net, count, H, W, false, net->out, fit ? &st : nullptr, s)) != ADMM_OK) return rc;
    if (fit) return ADMM_OK;         // the last layer has written the starts
    split_start_ptrs_kernel<<<grid, 256, 0, s>>>(net->out, g_ws.scales[0], g_ws.scales[1], g_ws.scales[2], P, hw);
    ++g_cnn_launches;
    CKC(cudaGetLastError());
    return ADMM_OK;
}
}  // namespace admm
