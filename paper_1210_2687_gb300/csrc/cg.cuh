// cg.cuh -- the Reeves-Sorel variants TV-CG and FA-CG (Sec. IV-C/IV-D,
// "Using the Reeves-Sorel technique").
//
// There the observation split is u1 = M A x with g1(u) = 1/2 ||y - u||^2 on
// the observed pixels (eq. H_1_analysis_sorel), and the x-step inverse
// (A^T M^T M A + gamma D^T D)^{-1} (TV) or (A^T M^T M A + gamma I)^{-1}
// (frame) is applied as C - C B^T (B C B^T - I)^{-1} B C (eqs. ReevesTV,
// reeves3), C the circulant inverse the column phase already applies and B
// the rows of A at the unobserved pixels U. The inner system takes one
// conjugate-gradient iteration per outer iteration, warm-started from the
// previous one (Sec. IV-B).
//
// The kernels carry the inner unknown as z = -xi (xi the paper's unknown),
// which solves the positive definite (I - B C B^T) z = B C r; CG takes the
// same steps on either sign. With r = A^T M^T zeta1 + w (w = gamma D^T delta
// or gamma P^T zeta2) one outer iteration is:
//   1. x~ = C (r + B^T z)            -- the column phase on the row DFTs of
//                                       zeta~ + i w, where zeta~ holds zeta1
//                                       on observed pixels and z on U (so
//                                       A^T zeta~ = A^T M^T zeta1 + B^T z)
//   2. s = B x~ - z                   -- the CG residual at the warm start
//                                       (cg_row_a, which also sends s + i 0
//                                       to the row DFTs for step 3)
//   3. v = C A^T s, A v               -- the column phase again
//   4. alpha = s.s / s.(s - B v)      -- the exact step along s (cg_row_b;
//                                       its last CTA divides)
//   5. x = x~ + alpha v, A x likewise, z += alpha s; then the observation
//      prox and dual update on the observed pixels (cg_obs), and the
//      regulariser side as for the MD methods (tv_tile for TV; the frame
//      analysis and synthesis tiles for the frame prior), which finishes
//      the iteration; the forward row DFTs of zeta~ + i w close it.
// Per-pixel planes (ProbDesc::cg): x~, A x~, v, A v, s, z.
#pragma once
#include "haar.cuh"
#include "variants.cuh"

namespace admm {

// Block sum of one compensated FP32 accumulator into thread 0 (FP64).
__device__ __forceinline__ double block_sum_comp(const CompSum& a, double* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float s = a.s, c = a.c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, o);
        c += __shfl_down_sync(0xffffffffu, c, o);
    }
    if (lane == 0) red[warp] = (double)s + (double)c;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < kThreads / 32; ++w) t += red[w];
    return t;
}

// ---------------------------------------------------------------------------
// step 2: inverse row DFTs -> x~, A x~; s = A x~ - z on U (0 elsewhere);
// forward row DFTs of s + i 0 -> Sb. Grid: (H / G, slots), G rows per CTA.
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(kThreads)
cg_row_a(const ProbDesc* __restrict__ probs, SlotTable sl, int H, int Wp, const float2* __restrict__ tw_g) {
    chain_wait();   // (launch chain: the predecessor's writes are visible)
    constexpr int FT = W / 8, G = kThreads / FT;
    const int pi = sl.map[blockIdx.y];
    if (pi < 0) return;
    const ProbDesc& P = probs[pi];
    if (P.ctl->active == 0) return;
    const int k = P.ctl->iter + 1;
    const bool cold = k == 1 && !P.warm;         // z = 0 at the start
    extern __shared__ __align__(16) float2 smem[];
    float2* buf = smem;
    float2* tw = buf + G * W;
    double* red = reinterpret_cast<double*>(tw + W);
    const int tid = threadIdx.x, g = tid / FT, t = tid % FT;
    const int q = blockIdx.x * G + g;
    const size_t n = (size_t)H * W;
    float* __restrict__ X = P.cg;
    float* __restrict__ AX = P.cg + n;
    float* __restrict__ Sv = P.cg + 4 * n;
    const float* __restrict__ Z = P.cg + 5 * n;
    const float* __restrict__ Y = P.ybar;
    // everything the CTA reads is requested before the transform: a load between
    // the stores below would wait for each of them in turn (eight latencies)
    float2 v[8];
    float yb[8], z[8];
    load_row_xax<W>(v, P.Sa + (size_t)q * Wp, t);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const size_t pix = (size_t)q * W + t + m * FT;
        yb[m] = Y[pix];
        z[m] = cold ? 0.f : Z[pix];
    }
    load_twiddles<W>(tw, tw_g, tid, kThreads);
    __syncthreads();
    float2* row = buf + g * W;
    fft_group<W, 1>(v, row, tw, t, g);
    CompSum ss;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const size_t pix = (size_t)q * W + t + m * FT;
        const float x = v[m].x, ax = v[m].y;
        const bool obs = is_observed(yb[m]);
        const float s = obs ? 0.f : ax - z[m];
        X[pix] = x;
        AX[pix] = ax;
        Sv[pix] = s;
        ss.add(s * s);
        v[m] = make_float2(s, 0.f);
    }
    fft_group<W, -1>(v, row, tw, t, g);
#pragma unroll
    for (int m = 0; m < 8; ++m) row[swz(t + m * FT)] = v[m];
    group_sync<W>(g);                // the split reads this group's row only
    store_split<W>(P.Sb + (size_t)q * Wp, row, t);
    const double tot = block_sum_comp(ss, red);
    if (tid == 0) P.cg_part[blockIdx.x] = tot;
}

// ---------------------------------------------------------------------------
// step 4: inverse row DFTs -> v = C A^T s, A v; the CTA's share of
// s.(s - A v) over U; the last CTA of the problem reduces both sums in a
// fixed order and sets alpha. Grid: (H / G, slots).
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(kThreads)
cg_row_b(const ProbDesc* __restrict__ probs, SlotTable sl, int H, int Wp, const float2* __restrict__ tw_g) {
    chain_wait();   // (launch chain: the predecessor's writes are visible)
    constexpr int FT = W / 8, G = kThreads / FT;
    const int pi = sl.map[blockIdx.y];
    if (pi < 0) return;
    const ProbDesc& P = probs[pi];
    ProbCtl* ctl = P.ctl;
    if (ctl->active == 0) return;
    extern __shared__ __align__(16) float2 smem[];
    float2* buf = smem;
    float2* tw = buf + G * W;
    double* red = reinterpret_cast<double*>(tw + W);
    __shared__ int s_last;
    const int tid = threadIdx.x, g = tid / FT, t = tid % FT;
    const int q = blockIdx.x * G + g;
    const int nrow = H / G;
    const size_t n = (size_t)H * W;
    float* __restrict__ V = P.cg + 2 * n;
    float* __restrict__ AV = P.cg + 3 * n;
    const float* __restrict__ Sv = P.cg + 4 * n;
    float2 v[8];
    float sv[8];                                  // 0 on observed pixels (requested before the transform)
    load_row_xax<W>(v, P.Sa + (size_t)q * Wp, t);
#pragma unroll
    for (int m = 0; m < 8; ++m) sv[m] = Sv[(size_t)q * W + t + m * FT];
    load_twiddles<W>(tw, tw_g, tid, kThreads);
    __syncthreads();
    fft_group<W, 1>(v, buf + g * W, tw, t, g);
    CompSum den;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const size_t pix = (size_t)q * W + t + m * FT;
        V[pix] = v[m].x;
        AV[pix] = v[m].y;
        den.add(sv[m] * (sv[m] - v[m].y));
    }
    const double tot = block_sum_comp(den, red);
    if (tid == 0) {
        P.cg_part[nrow + blockIdx.x] = tot;
        __threadfence();
        s_last = atomicAdd(&ctl->cg_arrive, 1u) == (unsigned)(nrow - 1);
    }
    __syncthreads();
    if (!s_last) return;
    // the last CTA: both sums over all row CTAs, each thread a fixed strided
    // share, then a fixed tree (reproducible)
    __threadfence();
    double a = 0.0, b = 0.0;
    for (int i = tid; i < nrow; i += kThreads) {
        a += __ldcg(P.cg_part + i);
        b += __ldcg(P.cg_part + nrow + i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    if (lane == 0) {
        red[warp] = a;
        red[kThreads / 32 + warp] = b;
    }
    __syncthreads();
    if (tid == 0) {
        double ta = 0.0, tb = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) {
            ta += red[w];
            tb += red[kThreads / 32 + w];
        }
        // s = 0 (nothing unobserved, or already solved): no step
        ctl->cg_alpha = (ta > 0.0 && tb > 0.0) ? (float)(ta / tb) : 0.f;
        ctl->cg_arrive = 0u;
    }
}

// ---------------------------------------------------------------------------
// step 5, observation side: x = x~ + alpha v, A x = A x~ + alpha A v; on
// observed pixels u1 = (y + mu1 (A x - d1)) / (1 + mu1), d1 <- d1 - (A x - u1)
// (prox of g1 = 1/2 ||y - u||^2 and Alg. 3 line 8 with M A); on U z += alpha s.
// Writes x and zeta~ (zeta1 = u1 + d1 on observed pixels, z on U) to the
// scratch planes, and the data-term, rel-x and d1 partial sums in the slots
// of the row kernels. Grid: (H / G, slots), the row kernels' layout.
// ---------------------------------------------------------------------------
template <int W>
__global__ void __launch_bounds__(kThreads)
cg_obs(const ProbDesc* __restrict__ probs, SlotTable sl, int H) {
    chain_wait();   // (launch chain: the predecessor's writes are visible)
    constexpr int FT = W / 8, G = kThreads / FT;
    const int pi = sl.map[blockIdx.y];
    if (pi < 0) return;
    const ProbDesc& P = probs[pi];
    if (P.ctl->active == 0) return;
    const int k = P.ctl->iter + 1;
    const bool first = k == 1;                   // x_prev = 0 (no earlier iterate)
    const bool cold = first && !P.warm;          // d1 = 0, z = 0
    const bool chk = is_check_iter(P, k), sprev = store_prev_iter(P, k), nobj = need_obj_iter(P, k);
    __shared__ float red[kThreads / 32 * 2 * kNumPartials];
    const int tid = threadIdx.x, g = tid / FT, t = tid % FT;
    const int q = blockIdx.x * G + g;
    const size_t n = (size_t)H * W;
    const float alpha = P.ctl->cg_alpha;
    const float* __restrict__ X = P.cg;
    const float* __restrict__ AX = P.cg + n;
    const float* __restrict__ V = P.cg + 2 * n;
    const float* __restrict__ AV = P.cg + 3 * n;
    const float* __restrict__ Sv = P.cg + 4 * n;
    float* __restrict__ Z = P.cg + 5 * n;
    float* __restrict__ xw = P.work;
    float* __restrict__ z1w = P.work + n;
    const float* __restrict__ Y = P.ybar;
    float* __restrict__ D1 = P.d1;
    float* __restrict__ XP = P.xprev;
    const float mu1 = P.mu1, inv1 = P.inv1pmu1;
    // all reads first (whatever the pixel needs of them): between the stores each
    // would wait its own latency
    float xv[8], axv[8], yv[8], dv[8], zv[8], pv8[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const size_t pix = (size_t)q * W + t + m * FT;
        xv[m] = fmaf(alpha, V[pix], X[pix]);
        axv[m] = fmaf(alpha, AV[pix], AX[pix]);
        yv[m] = Y[pix];
        dv[m] = cold ? 0.f : D1[pix];
        zv[m] = fmaf(alpha, Sv[pix], cold ? 0.f : Z[pix]);
        pv8[m] = (chk && !first) ? XP[pix] : 0.f;
    }
    CompSum s_data, s_xx, s_dxx, s_pr;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        const size_t pix = (size_t)q * W + t + m * FT;
        const float x = xv[m], ax = axv[m], yb = yv[m];
        float z1 = zv[m], nd1 = 0.f;
        if (is_observed(yb)) {
            const float dd1 = dv[m];
            const float u1 = fmaf(mu1, ax - dd1, yb) * inv1;
            nd1 = dd1 - (ax - u1);
            z1 = u1 + nd1;
            if (nobj) {
                const float e = ax - yb;
                s_data.add(0.5f * e * e);
                const float e1 = nd1 - dd1;
                s_pr.add(e1 * e1);
            }
        } else {
            Z[pix] = z1;
        }
        D1[pix] = nd1;
        xw[pix] = x;
        z1w[pix] = z1;
        if (chk) {
            const float dx = x - pv8[m];
            s_dxx.add(dx * dx);
            s_xx.add(x * x);
        }
        if (sprev) XP[pix] = x;
    }
    if (nobj || chk) {
        const CompSum acc[kNumPartials] = {s_data, CompSum(), s_xx, s_dxx, s_pr};
        double pv[kNumPartials];
        block_reduce_comp(acc, red, pv);
        if (tid == 0) {
#pragma unroll
            for (int j = 0; j < kNumPartials; ++j) P.partials[blockIdx.x * kNumPartials + j] = pv[j];
        }
    }
}

// ---------------------------------------------------------------------------
// TV regulariser side on a 32 x 32 tile (Alg. 3 lines 9-11 and lines 3-5 of
// the next iteration), for TV-CG and for TV-MD on domains whose sides are
// not both powers of two: D x with forward periodic differences, vector-soft
// (ANISO: eq. soft per component) with tau = lambda / mu2, d2 <- d2 -
// (D x - u2), delta = u2 + d2 and w = gamma (Dh^T delta_h + Dv^T delta_v).
// w at a pixel needs delta one column left and one row up, so the tile
// recomputes delta on that halo from x (one more row and column of x) and
// the previous d2 (double-buffered by iteration parity, so a neighbour's halo
// always sees the old d2). Finishes the iteration. Grid: (tiles, slots).
// H and W are multiples of 32 (not necessarily powers of two).
//
// Bound by memory latency (28 B per pixel, a few tiles per SM): a thread owns
// four adjacent pixels of row tid / 8 and requests everything it needs, 16
// bytes at a time, before anything else; the left column's delta_h comes by
// shuffle, delta_v goes through shared memory once, and eight threads and one
// warp take the row above and the column left of the tile as well. 8 x 384^2:
// 14.3 -> 12.3 us per launch.
// ---------------------------------------------------------------------------
constexpr int kCgTile = 32;
template <bool ANISO = false>
__global__ void __launch_bounds__(kThreads, 4)
tv_tile(const ProbDesc* __restrict__ probs, SlotTable sl, int H, int W, int n_row_ctas,
        int* __restrict__ n_active) {
    chain_wait();   // (launch chain: the predecessor's writes are visible)
    constexpr int T = kCgTile;
    static_assert(T * T == 4 * kThreads, "four pixels per thread");
    const int pi = sl.map[blockIdx.y];
    if (pi < 0) return;
    const ProbDesc& P = probs[pi];
    if (P.ctl->active == 0) return;
    const int k = P.ctl->iter + 1;
    const bool first = k == 1 && !P.warm;        // d2 = 0 (cold start)
    const bool chk = is_check_iter(P, k), nobj = need_obj_iter(P, k);
    __shared__ __align__(16) float dvs[(T + 1) * T];   // delta_v on rows R0-1 .. R0+T-1
    __shared__ float dhs[T];                     // delta_h on column C0-1
    __shared__ float red[kThreads / 32 * 2 * kNumPartials];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles_x = W / T;
    const int R0 = (blockIdx.x / tiles_x) * T, C0 = (blockIdx.x % tiles_x) * T;
    const size_t n = (size_t)H * W;
    const float* __restrict__ xw = P.work;
    float* __restrict__ ww = P.work + 2 * n;
    const float2* __restrict__ d2in = reinterpret_cast<const float2*>(P.d2 + ((k + 1) & 1) * P.d2_stride);
    float2* __restrict__ d2out = reinterpret_cast<float2*>(P.d2 + (k & 1) * P.d2_stride);
    const float tau = P.tau, gam = P.gamma;
    // four adjacent pixels (r, c .. c + 3): x, x below, x right of the last one, d2
    struct Quad {
        float x[5], xd[4], dh[4], dv[4];
    };
    auto load = [&](int r, int c) {
        Quad v;
        const int rd = r + 1 == H ? 0 : r + 1, cr = c + 4 == W ? 0 : c + 4;
        const float4 a = *reinterpret_cast<const float4*>(xw + (size_t)r * W + c);
        const float4 b = *reinterpret_cast<const float4*>(xw + (size_t)rd * W + c);
        v.x[4] = xw[(size_t)r * W + cr];
        float4 d0 = make_float4(0.f, 0.f, 0.f, 0.f), d1 = d0;
        if (!first) {
            d0 = *reinterpret_cast<const float4*>(d2in + (size_t)r * W + c);
            d1 = *reinterpret_cast<const float4*>(d2in + (size_t)r * W + c + 2);
        }
        v.x[0] = a.x; v.x[1] = a.y; v.x[2] = a.z; v.x[3] = a.w;
        v.xd[0] = b.x; v.xd[1] = b.y; v.xd[2] = b.z; v.xd[3] = b.w;
        v.dh[0] = d0.x; v.dv[0] = d0.y; v.dh[1] = d0.z; v.dv[1] = d0.w;
        v.dh[2] = d1.x; v.dv[2] = d1.y; v.dh[3] = d1.z; v.dv[3] = d1.w;
        return v;
    };
    // u2 = prox(D x - d2), d2 <- d2 - (D x - u2), delta = u2 + d2 of one pixel
    auto step = [&](float gh, float gv, float odh, float odv, float& ndh, float& ndv, float& eh, float& ev) {
        float uh, uv;
        tv_prox(gh - odh, gv - odv, tau, ANISO, uh, uv);
        ndh = odh - (gh - uh);
        ndv = odv - (gv - uv);
        eh = uh + ndh;
        ev = uv + ndv;
    };
    const int orow = tid >> 3, ocol = 4 * (tid & 7);
    const Quad own = load(R0 + orow, C0 + ocol);
    // the halo: threads 0..7 the row above, warp 1 (one row per lane) the column left
    Quad up = {};
    float lx = 0.f, lxr = 0.f, lxd = 0.f;
    float2 ld = make_float2(0.f, 0.f);
    if (tid < 8) up = load(R0 == 0 ? H - 1 : R0 - 1, C0 + ocol);
    if (warp == 1) {
        const int r = R0 + lane, rd = r + 1 == H ? 0 : r + 1, c = C0 == 0 ? W - 1 : C0 - 1;
        lx = xw[(size_t)r * W + c];
        lxr = xw[(size_t)r * W + C0];
        lxd = xw[(size_t)rd * W + c];
        if (!first) ld = d2in[(size_t)r * W + c];
    }
    CompSum tvs, prs;
    float dh[4], dv[4], nh[4], nv[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float gh = own.x[e + 1] - own.x[e], gv = own.xd[e] - own.x[e];
        step(gh, gv, own.dh[e], own.dv[e], nh[e], nv[e], dh[e], dv[e]);
        if (nobj) {
            tvs.add(tv_norm(gh, gv, ANISO));
            const float eh = nh[e] - own.dh[e], ev = nv[e] - own.dv[e];
            prs.add(fmaf(eh, eh, ev * ev));
        }
    }
    *reinterpret_cast<float4*>(dvs + (orow + 1) * T + ocol) = make_float4(dv[0], dv[1], dv[2], dv[3]);
    if (tid < 8) {
        float a, b, h, v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            step(up.x[e + 1] - up.x[e], up.xd[e] - up.x[e], up.dh[e], up.dv[e], a, b, h, v[e]);
        *reinterpret_cast<float4*>(dvs + ocol) = make_float4(v[0], v[1], v[2], v[3]);
    }
    if (warp == 1) {
        float a, b, h, v;
        step(lxr - lx, lxd - lx, ld.x, ld.y, a, b, h, v);
        dhs[lane] = h;
    }
    const size_t pix = (size_t)(R0 + orow) * W + (C0 + ocol);
    *reinterpret_cast<float4*>(d2out + pix) = make_float4(nh[0], nv[0], nh[1], nv[1]);
    *reinterpret_cast<float4*>(d2out + pix + 2) = make_float4(nh[2], nv[2], nh[3], nv[3]);
    const float sh = __shfl_up_sync(0xffffffffu, dh[3], 1);
    __syncthreads();
    const float4 u = *reinterpret_cast<const float4*>(dvs + orow * T + ocol);
    const float left = (tid & 7) == 0 ? dhs[orow] : sh;
    *reinterpret_cast<float4*>(ww + pix) =
        make_float4(gam * ((left - dh[0]) + (u.x - dv[0])), gam * ((dh[0] - dh[1]) + (u.y - dv[1])),
                    gam * ((dh[1] - dh[2]) + (u.z - dv[2])), gam * ((dh[2] - dh[3]) + (u.w - dv[3])));
    double pv[kNumPartials] = {0.0};
    if (nobj || chk) {
        const CompSum acc[kNumPartials] = {CompSum(), tvs, CompSum(), CompSum(), prs};
        block_reduce_comp(acc, red, pv);
    }
    finish_iteration<kThreads>(P, k, chk, nobj, pv, n_active, n_row_ctas + blockIdx.x, probs, sl);
}

inline int cg_num_tiles(int H, int W) { return (H / kCgTile) * (W / kCgTile); }

// One TV-CG (tv = true) or FA-CG iteration of a lane: the two column phases
// (col_fn) and the row-side kernels, as a launch chain (cg.cu).
cudaError_t launch_cg_iteration(int W, int H, int Wc, int Wp, const ProbDesc* d, SlotTable sl, int count,
                                int levels, bool tv, ColLaunchFn col_fn, const float2* tw, int* n_active,
                                cudaStream_t s);

}  // namespace admm
