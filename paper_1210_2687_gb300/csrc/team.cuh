// team.cuh -- TV-MD iterations of a small image on a team of CTAs, many
// iterations per launch.
//
// An image of at most 256 x 256 fills a few SMs. Run as one column-phase and
// one row-phase launch per iteration (kernels.cuh) it is bound by latency:
// launch boundaries, the strip's serial walk, and every CTA fetching its
// descriptor, twiddles, spectra and duals again. Here a team of C CTAs keeps
// the image for the whole launch: CTA j the rows [j R, (j + 1) R), R = H / C,
// and NC columns of the half spectrum. The duals stay in registers, M^T y,
// x_prev, Lambda and K in shared memory; only the spectra change hands, and a
// barrier of the team takes the place of each launch boundary.
//
// Per iteration:
//   column phase   the CTA's columns, one group of H/8 threads per signal:
//                  forward DFTs of zeta1 and w, x^ = K (conj(Lambda) Z1^ + W^),
//                  (A x)^ = Lambda x^, inverse DFTs
//   barrier
//   row phase      one row per group of W/8 threads, all rows at once, a pixel's
//                  state with the thread that transforms it: inverse DFT, mask
//                  prox and d1 (eq. new_line, Alg. 3 line 8), differences, prox
//                  and d2 (lines 9-11), w, forward DFT, split into half spectra.
//                  The rows next to the CTA's own are transformed here too (x
//                  below; delta_v above, with its own copy of that row's d2).
//   barrier
// The arithmetic of each step is that of col_phase and row_phase_tv in any of
// their configurations, so a problem solved alone here and in a large batch
// there has the same iterates bit for bit (the objective and the relative changes
// are summed in another order).
//
// Stop rule: on iterations that evaluate it every CTA writes its partial sums,
// and after the barrier one warp of every CTA adds all CTAs' in the same order
// and takes the same decision, while the others already transform the next
// iteration's columns; nothing of that is stored if the decision is to stop.
//
// Up to 128 x 256 pixels the team is a thread-block cluster (8 or 16 CTAs): the
// spectra go to the CTA that needs them through distributed shared memory, and
// the hardware's cluster barrier costs 0.5 us where storing to L2, a barrier and
// loading cost 1.9 us (64 x 64: 6.9 us per iteration through L2). That barrier
// has no time limit; nothing else in a cluster's team waits. A 256 x 256 image
// needs more SMs than a cluster has: its transforms alone take 7 us on 16 SMs
// (15.8 us per iteration as a cluster), so there 64 CTAs, launched cooperatively,
// exchange through L2, and their barrier's waits are bounded.
// Whole calls, against the general kernels (two launches per iteration):
// 64 x 64, 200 iterations 668 against 2488 us; 256 x 256 with the objective
// evaluated in each of 80 iterations 812 against 1620 us.
#pragma once
#include <type_traits>

#include "kernels.cuh"

namespace admm {

constexpr int kMaxTeam = 64;          // CTAs per image (the partial sums of a plan have room for as many)
constexpr int kTeamSteps = 512;       // iterations per launch: a few milliseconds at 256 x 256

// One image over C CTAs. DSM: the CTAs are a thread-block cluster; the half
// spectra go straight to the CTA that reads them (distributed shared memory)
// and the hardware cluster barrier separates the phases. Otherwise they go
// through Sa and Sb (in L2) and a counter in the control block is the barrier
// (cooperative launch, bounded waits).
template <int H, int W>
struct TeamCfg {
    static constexpr bool DSM = H * W <= 128 * 256;
    static constexpr int C = DSM ? (H >= 128 ? 16 : 8) : 64;
    static constexpr int R = H / C;                     // rows per CTA
    static constexpr int GR = R + 2;                    // rows transformed
    static constexpr int FT = W / 8, FH = H / 8;        // threads per row / column transform
    static constexpr int Wc = W / 2 + 1;
    static constexpr int NC = ((Wc + C - 1) / C) | 1;   // columns per CTA (odd: conflict-free columns of the tile)
    static constexpr int NTR = GR * FT, NTC = NC * 2 * FH;   // threads of the row / column phase
    // + one warp that reduces and decides
    static constexpr int NT = ((NTR > NTC ? NTR : NTC) + 31) / 32 * 32 + 32;
    static_assert(FT <= 32 && FH <= 32 && NT <= 1024 && C <= kMaxTeam, "small images");
    // shared memory: the column tile and the row spectra (written by other CTAs
    // while this one is in the other phase, so apart from the scratch), the
    // phases' scratch in turn, then what stays: Lambda, K, M^T y, x_prev, twiddles
    static constexpr size_t TILE = (size_t)H * NC * sizeof(float4);
    static constexpr size_t SPEC = (size_t)GR * Wc * sizeof(float4);
    static constexpr size_t CSCR = (size_t)NC * 2 * H * sizeof(float2);
    static constexpr size_t RSCR = (size_t)GR * W * sizeof(float2) + (size_t)(GR + R + 1) * W * sizeof(float);
    static constexpr size_t SCR = ((CSCR > RSCR ? CSCR : RSCR) + 15) / 16 * 16;
    static constexpr size_t LK = (size_t)NC * H * (sizeof(float2) + sizeof(float));
    static constexpr size_t PIX = (size_t)2 * R * W * sizeof(float);
    static constexpr size_t SMEM = TILE + SPEC + SCR + LK + PIX + (size_t)(W + H) * sizeof(float2);
};

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// this address of shared memory in the cluster's CTA `rank`
__device__ __forceinline__ uint32_t remote(const void* p, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t a, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_remote2(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// Grid: C x slots (DSM: clusters of C). Runs up to max_steps iterations of the
// slot's problem.
template <int H, int W, bool ANISO>
__global__ void __launch_bounds__((TeamCfg<H, W>::NT))
tv_team(const ProbDesc* __restrict__ probs, SlotTable sl, int Wp, const float2* __restrict__ tw_g,
        int* __restrict__ n_active, int max_steps) {
    using C = TeamCfg<H, W>;
    constexpr int R = C::R, FT = C::FT, FH = C::FH, NC = C::NC, Wc = C::Wc, NWARP = C::NT / 32;
    constexpr bool DSM = C::DSM;
    const int slot = blockIdx.x / C::C, rank = blockIdx.x % C::C;
    const int pi = sl.map[slot];
    if (pi < 0) return;                              // (the same for the whole team)
    const ProbDesc& P = probs[pi];
    ProbCtl* const ctl = P.ctl;
    if (ctl->active == 0) return;
    if (ctl->status == kStatusTimeout) {             // (a wait of another CTA ran out at the end of the last launch)
        if (rank == 0 && threadIdx.x == 0) {
            ctl->active = 0;
            ctl->t_done = device_clock_ns();
            atomicSub(n_active, 1);
        }
        return;
    }
    extern __shared__ __align__(16) unsigned char cl_raw[];
    float4* tile = reinterpret_cast<float4*>(cl_raw);                      // [H][NC]
    float4* spec = reinterpret_cast<float4*>(cl_raw + C::TILE);            // [GR][Wc]
    unsigned char* scr = cl_raw + C::TILE + C::SPEC;
    float2* cscr = reinterpret_cast<float2*>(scr);                         // [NC][2][H]
    float2* rscr = reinterpret_cast<float2*>(scr);                         // [GR][W]
    float* xs = reinterpret_cast<float*>(rscr + C::GR * W);                // [GR][W]
    float* dvs = xs + C::GR * W;                                           // [R + 1][W]
    float2* lam_s = reinterpret_cast<float2*>(scr + C::SCR);               // [NC][H]
    float* k_s = reinterpret_cast<float*>(lam_s + NC * H);                 // [NC][H]
    float* yb_s = k_s + NC * H;                                            // [R][W]
    float* xp_s = yb_s + R * W;                                            // [R][W]
    float2* tww = reinterpret_cast<float2*>(xp_s + R * W);
    float2* twh = tww + W;
    __shared__ float red[NWARP * 2 * kNumPartials];
    __shared__ double part_s[DSM ? C::C * kNumPartials : 1];
    __shared__ int s_stop;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r0 = rank * R, c0 = rank * NC;
    const int ncol = max(0, min(NC, Wc - c0));       // columns of this CTA
    // row role: group i transforms image row r0 - 1 + i; its thread t owns columns t + m FT
    const int i = tid / FT, t = tid % FT;
    const bool rowthr = i < C::GR, owned = i >= 1 && i <= R, tvrow = i <= R;
    const int q = (r0 - 1 + i + H) % H;
    // column role: the groups 2 g and 2 g + 1 transform the two signals of column c0 + g
    const int gg = tid / FH, s = tid % FH, g = gg >> 1, sig = gg & 1;
    const bool colthr = g < ncol;
    const bool service = warp == NWARP - 1;

    const int k0 = ctl->iter;
    const bool start = k0 == 0;
    const bool zero = start && !P.warm;              // u0 = d0 = 0
    const int kend = min(P.max_iters, k0 + max_steps);
    // stop rule state (the same in every CTA)
    double obj_prev = ctl->obj_prev, obj = ctl->obj, rel_x = ctl->rel_x, rel_obj = ctl->rel_obj,
           primal_res = ctl->primal_res;
    int have_obj = ctl->have_obj, status = ctl->status, conv = 0;

    // what the loop reads of the descriptor, by value: the barriers' acquire would
    // have every access to it go back to L2
    const float tau = P.tau, gam = P.gamma, mu1 = P.mu1, inv1 = P.inv1pmu1, lam = P.lam;
    float4* const Sa = P.Sa;
    float4* const Sb = P.Sb;
    double* const partials = P.partials;
    const int rule = P.stop, max_iters = P.max_iters, every = P.check_every, warm = P.warm;
    const double tol = P.tol;

    load_twiddles<W>(tww, tw_g, tid, C::NT);
    load_twiddles<H>(twh, tw_g, tid, C::NT);
    for (int e = tid; e < ncol * H; e += C::NT) {
        lam_s[e] = P.lamT[(size_t)c0 * H + e];
        k_s[e] = P.kT[(size_t)c0 * H + e];
    }
    for (int e = tid; e < R * W; e += C::NT) {
        yb_s[e] = P.ybar[(size_t)r0 * W + e];
        xp_s[e] = start ? 0.f : P.xprev[(size_t)r0 * W + e];
    }
    if (DSM && !zero)
        for (int e = tid; e < H * ncol; e += C::NT)
            tile[e / ncol * NC + e % ncol] = Sb[(size_t)(e / ncol) * Wp + c0 + e % ncol];
    float d1[8], dh[8], dv[8];                       // duals of the owned pixels (dh, dv also of the row above)
    {
        // iteration k reads d2 buffer (k + 1) & 1
        const float2* __restrict__ d2in = reinterpret_cast<const float2*>(P.d2 + (k0 & 1) * P.d2_stride);
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const size_t pix = (size_t)q * W + t + m * FT;
            const float2 v = (tvrow && !zero) ? d2in[pix] : make_float2(0.f, 0.f);
            dh[m] = v.x;
            dv[m] = v.y;
            d1[m] = (owned && !zero) ? P.d1[pix] : 0.f;
        }
    }
    // Barrier of the team. Without clusters: bar counts the arrivals of the whole
    // solve; false if a wait ran out (about a second).
    unsigned target = ctl->team_base;
    bool first_bar = true;
    // (test hook: the last CTA's wait at the launch's second barrier counts as one that ran out)
    const bool gives_up = !DSM && P.test_stall && rank == C::C - 1;
    auto barrier = [&]() -> bool {
        if constexpr (DSM) {
            cluster_barrier();
            return true;
        } else {
            __shared__ int s_ok;
            target += C::C;
            __syncthreads();
            if (tid == 0) {
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->team_bar) : "memory");
                // bounded: about a second; ten at the first barrier, where CTAs may wait for
                // other work to leave its SMs. The clock is read every 256 polls.
                unsigned long long t0 = 0;
                const unsigned long long limit = first_bar ? 10000000000ull : 1000000000ull;
                int good = gives_up && !first_bar ? 0 : 1;
                for (unsigned n = 1;; ++n) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->team_bar) : "memory");
                    if ((int)(v - target) >= 0) break;
                    if ((n & 255u) == 0) {
                        const unsigned long long now = device_clock_ns();
                        if (t0 == 0) t0 = now;
                        if (now - t0 > limit) {
                            good = 0;
                            break;
                        }
                    }
                }
                s_ok = good;
                first_bar = false;
            }
            __syncthreads();
            return s_ok != 0;
        }
    };
    if constexpr (DSM) cluster_barrier();            // every CTA has started: its shared memory may be written
    else __syncthreads();

    // (service warp) all CTAs' partial sums of iteration k in rank order, the
    // stop rule as in finish_iteration; every lane holds the result
    auto decide = [&](int k, bool chk, bool nobj) -> bool {
        // six lanes per sum, each every sixth CTA's share, then the six in a fixed order
        constexpr int PARTS = 6;
        const int js = lane % kNumPartials, jp = lane / kNumPartials;
        double val[(C::C + PARTS - 1) / PARTS];
#pragma unroll
        for (int j = 0; j < (C::C + PARTS - 1) / PARTS; ++j) {
            const int c = j * PARTS + jp;
            val[j] = (jp < PARTS && c < C::C) ? (DSM ? part_s[c * kNumPartials + js] : __ldcg(partials + c * kNumPartials + js))
                                              : 0.0;
        }
        double acc = 0.0;
#pragma unroll
        for (int j = 0; j < (C::C + PARTS - 1) / PARTS; ++j) acc += val[j];
        acc += __shfl_down_sync(0xffffffffu, acc, 3 * kNumPartials);
        acc = (acc + __shfl_down_sync(0xffffffffu, acc, kNumPartials)) + __shfl_down_sync(0xffffffffu, acc, 2 * kNumPartials);
        double a[kNumPartials];
#pragma unroll
        for (int j = 0; j < kNumPartials; ++j) a[j] = __shfl_sync(0xffffffffu, acc, j);
        bool done = status != 0, cv = false;
        if (nobj) {
            const double f = a[0] + (double)lam * a[1];
            if (!isfinite(f)) {
                status = kStatusNonFinite;
                done = true;
            }
            if (rule == kStopRelObj && have_obj) {
                rel_obj = (f != 0.0) ? fabs(f - obj_prev) / fabs(f) : INFINITY;
                if (rel_obj < tol) cv = true;
            }
            obj_prev = obj = f;
            have_obj = 1;
            primal_res = sqrt(fmax(a[4], 0.0));
        }
        if (chk) {
            if (!isfinite(a[2]) || !isfinite(a[3])) {
                status = kStatusNonFinite;
                done = true;
            }
            rel_x = (a[2] > 0.0) ? sqrt(a[3] / a[2]) : INFINITY;
            if (rel_x < tol) cv = true;
        }
        if (cv && !done) conv = 1;
        return cv || done || k >= max_iters;
    };
    // both signals of a column are transformed: their groups wait for each other
    auto pair_sync = [&]() {
        if constexpr (2 * FH <= 32) {
            constexpr unsigned lanes = 2 * FH == 32 ? 0xffffffffu : ((1u << (2 * FH)) - 1u);
            __syncwarp(lanes << ((2 * g * FH) & 31));
        } else {
            asm volatile("bar.sync %0, %1;\n" ::"r"(1 + g), "n"(2 * FH) : "memory");
        }
    };

    int k = k0;                      // iterations done
    bool pend = false, pchk = false, pnobj = false, stop = false;   // a decision of iteration k is due
    bool alive = true;               // no wait has run out
    while (k < kend) {
        const bool cold = k == 0 && zero;
        // ---- column phase of iteration k + 1 ----
        if (cold) {
            // the right-hand side is zero, so x1 = 0
            if constexpr (DSM) {
                for (int e = tid; e < C::GR * Wc; e += C::NT) spec[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                for (int e = tid; e < H * ncol; e += C::NT)
                    Sa[(size_t)(e / ncol) * Wp + c0 + e % ncol] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        } else {
            if (service) {
                if (pend) {
                    stop = decide(k, pchk, pnobj);
                    if (lane == 0) s_stop = stop;
                }
            } else if constexpr (!DSM) {
                for (int e = tid; e < H * ncol; e += C::NT - 32) {
                    const int r = e / ncol, c = e - r * ncol;
                    cp_async16(tile + r * NC + c, Sb + (size_t)r * Wp + c0 + c);
                }
                cp_async_commit();
                cp_async_wait<0>();
                asm volatile("bar.sync 15, %0;\n" ::"n"(C::NT - 32) : "memory");   // (all warps but the deciding one)
            }
            float2 v[8];
            if (colthr) {
                const float2* in = reinterpret_cast<const float2*>(tile) + sig;
#pragma unroll
                for (int m = 0; m < 8; ++m) v[m] = in[2 * ((s + m * FH) * NC + g)];
                float2* own = cscr + gg * H;
                const float2* other = cscr + (gg ^ 1) * H;
                fft_group<H, -1>(v, own, twh, s, gg);
#pragma unroll
                for (int m = 0; m < 8; ++m) own[swz(s + m * FH)] = v[m];
                pair_sync();
                float2 p[8];
#pragma unroll
                for (int m = 0; m < 8; ++m) p[m] = other[swz(s + m * FH)];
                pair_sync();                         // the buffers may be written again
                const bool warm0 = k == 0 && warm == 1;          // the first x-step returns x0
                const float inv_hw = 1.0f / (float)(H * W);
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    // x^ = K (conj(Lambda) Z1^ + W^);  (A x)^ = Lambda x^
                    const float2 L = lam_s[g * H + s + m * FH];
                    const float2 z = sig ? p[m] : v[m], w = sig ? v[m] : p[m];
                    const float2 xh = warm0 ? inv_hw * z : k_s[g * H + s + m * FH] * (cmulc(z, L) + w);
                    v[m] = sig ? cmul(L, xh) : xh;
                }
                fft_group<H, 1>(v, own, twh, s, gg);
            }
            if (pend) {
                __syncthreads();
                if (s_stop) break;
            }
            if constexpr (DSM) {
                if (colthr) {
                    // to the CTA that owns the row, and to the neighbour that has it as its halo
                    const uint32_t off = (uint32_t)((c0 + g) * 16 + sig * 8);
                    static_assert(FH % R == 0, "a thread's rows lie alike in their CTAs");
                    const int ri = s % R + 1;
                    const float4* const dst = spec + ri * Wc;
#pragma unroll
                    for (int m = 0; m < 8; ++m) st_remote2(remote(dst, (s + m * FH) / R) + off, v[m]);
                    if (ri == 1 || ri == R) {
                        const float4* const halo = ri == 1 ? spec + (R + 1) * Wc : spec;
                        const int d = ri == 1 ? C::C - 1 : 1;
#pragma unroll
                        for (int m = 0; m < 8; ++m)
                            st_remote2(remote(halo, ((s + m * FH) / R + d) % C::C) + off, v[m]);
                    }
                }
            } else {
                if (colthr) {
                    float2* out = reinterpret_cast<float2*>(tile) + sig;
#pragma unroll
                    for (int m = 0; m < 8; ++m)      // (over the entries this thread has read)
                        out[2 * ((s + m * FH) * NC + g)] = v[m];
                }
                __syncthreads();
                for (int e = tid; e < H * ncol; e += C::NT) {
                    const int r = e / ncol, c = e - r * ncol;
                    Sa[(size_t)r * Wp + c0 + c] = tile[r * NC + c];
                }
            }
        }
        pend = false;
        if (!barrier()) {
            alive = false;
            break;
        }
        // ---- row phase of iteration k + 1 ----
        ++k;
        const bool first = k == 1;
        const bool relx = rule == kStopRelX;             // (is_check_iter, store_prev_iter, need_obj_iter)
        const bool chk = relx && (k % every == 0 || k == max_iters);
        const bool sprev = relx && ((k + 1) % every == 0 || k + 1 == max_iters);
        const bool nobj = rule == kStopRelObj || chk || k == max_iters;
        if constexpr (!DSM) {
            for (int e = tid; e < C::GR * Wc; e += C::NT) {
                const int r = e / Wc, c = e - r * Wc;
                cp_async16(spec + e, Sa + (size_t)((r0 - 1 + r + H) % H) * Wp + c);
            }
            cp_async_commit();
            cp_async_wait<0>();
            __syncthreads();
        }
        float2 v[8] = {};
        float ddh[8], ddv[8];                        // delta = u2 + d2
        // STATS: the iteration evaluates the objective (a check iteration does, too);
        // two bodies, each free of branches between its eight pixels
        auto row_phase = [&](auto stats) {
            constexpr bool STATS = decltype(stats)::value;
            CompSum s_data, s_reg, s_xx, s_dxx, s_pr;
            if (rowthr) {
                load_row_xax<W>(v, spec + i * Wc, t);
                fft_group<W, 1>(v, rscr + i * W, tww, t, i);
#pragma unroll
                for (int m = 0; m < 8; ++m) xs[i * W + t + m * FT] = v[m].x;
                if (owned) {
                    // u1 = (M^T M + mu1 I)^{-1} (M^T y + mu1 (A x - d1)); d1 <- d1 - (A x - u1); zeta1 = u1 + d1
#pragma unroll
                    for (int m = 0; m < 8; ++m) {
                        const int o = (i - 1) * W + t + m * FT;
                        const float x = v[m].x, ax = v[m].y, yb = yb_s[o], s1 = ax - d1[m];
                        const bool obs = is_observed(yb);
                        const float u1 = obs ? fmaf(mu1, s1, yb) * inv1 : s1;
                        const float nd1 = d1[m] - (ax - u1);
                        if constexpr (STATS) {
                            // (the sums of x are read on check iterations only)
                            const float e = obs ? ax - yb : 0.f, e1 = nd1 - d1[m];
                            const float dx = first ? x : x - xp_s[o];
                            s_data.add(0.5f * e * e);
                            s_pr.add(e1 * e1);
                            s_dxx.add(dx * dx);
                            s_xx.add(x * x);
                        }
                        d1[m] = nd1;
                        v[m].y = u1 + nd1;
                    }
                    if (sprev) {
#pragma unroll
                        for (int m = 0; m < 8; ++m) xp_s[(i - 1) * W + t + m * FT] = v[m].x;
                    }
                }
            }
            __syncthreads();                         // x of every row
            // differences, prox, d2 (every thread: the shuffles are by whole warps)
            float xr[8];
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                // right neighbour: the next lane of the group, its first lane's next column block at the end
                const float a = __shfl_down_sync(0xffffffffu, v[m].x, 1, FT);
                const float b = __shfl_sync(0xffffffffu, v[(m + 1) & 7].x, 0, FT);
                xr[m] = t == FT - 1 ? b : a;
            }
            const int id = tvrow ? i : 0;            // (other threads compute row 0's again and drop it)
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const float x = v[m].x, xd = xs[(id + 1) * W + t + m * FT];
                const float gh = xr[m] - x, gv = xd - x;
                const float sh = gh - dh[m], sv = gv - dv[m];
                float nh, nv;
                tv_split(sh, sv, tau, ANISO, nh, nv, ddh[m], ddv[m]);
                if constexpr (STATS) {
                    const float eh = nh - dh[m], ev = nv - dv[m];
                    s_reg.add(owned ? tv_norm(gh, gv, ANISO) : 0.f);
                    s_pr.add(owned ? fmaf(eh, eh, ev * ev) : 0.f);
                }
                dh[m] = nh;
                dv[m] = nv;
            }
            if (i < R) {
#pragma unroll
                for (int m = 0; m < 8; ++m) dvs[i * W + t + m * FT] = ddv[m];
            }
            if constexpr (STATS) {
                // warp sums of the running sums and of their compensation terms
                const CompSum acc[kNumPartials] = {s_data, s_reg, s_xx, s_dxx, s_pr};
#pragma unroll
                for (int j = 0; j < kNumPartials; ++j) {
                    float a = acc[j].s, b = acc[j].c;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        a += __shfl_down_sync(0xffffffffu, a, o);
                        b += __shfl_down_sync(0xffffffffu, b, o);
                    }
                    if (lane == 0) {
                        red[warp * 2 * kNumPartials + j] = a;
                        red[warp * 2 * kNumPartials + kNumPartials + j] = b;
                    }
                }
            }
        };
        if (nobj) row_phase(std::true_type());
        else row_phase(std::false_type());
        __syncthreads();                             // delta_v of every row, the warp sums
        if (service && (nobj || chk)) {
            double acc = 0.0;
            if (lane < 2 * kNumPartials)
                for (int w = 0; w < NWARP; ++w) acc += (double)red[w * 2 * kNumPartials + lane];
            const double tot = acc + __shfl_down_sync(0xffffffffu, acc, kNumPartials);
            if constexpr (DSM) {
                if (lane < kNumPartials)
                    for (int j = 0; j < C::C; ++j) st_remote(remote(part_s + rank * kNumPartials + lane, j), tot);
            } else {
                if (lane < kNumPartials) partials[rank * kNumPartials + lane] = tot;
            }
        }
        float dl[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const float a = __shfl_up_sync(0xffffffffu, ddh[m], 1, FT);
            const float b = __shfl_sync(0xffffffffu, ddh[(m + 7) & 7], FT - 1, FT);
            dl[m] = t == 0 ? b : a;
        }
        if (owned) {
            // w = gamma (Dh^T delta_h + Dv^T delta_v); p = zeta1 + i w
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const float up = dvs[(i - 1) * W + t + m * FT];
                // (rounded product: it must not be contracted into the transform's sums)
                v[m] = make_float2(v[m].y, __fmul_rn(gam, (dl[m] - ddh[m]) + (up - ddv[m])));
            }
            float2* row = rscr + i * W;
            fft_group<W, -1>(v, row, tww, t, i);
#pragma unroll
            for (int m = 0; m < 8; ++m) row[swz(t + m * FT)] = v[m];
            group_sync<W>(i);
            if constexpr (DSM) {
                // (as store_split) to the CTA that owns the column
#pragma unroll
                for (int m = 0; m <= 4; ++m) {
                    const int kc = t + m * FT;
                    if (kc > W / 2) break;
                    const float2 pk = row[swz(kc)];
                    const float2 pn = row[swz((W - kc) & (W - 1))];
                    const float2 a = 0.5f * make_float2(pk.x + pn.x, pk.y - pn.y);
                    const float2 dd = make_float2(pk.x - pn.x, pk.y + pn.y);
                    st_remote(remote(tile + q * NC + kc % NC, kc / NC), make_float4(a.x, a.y, 0.5f * dd.y, -0.5f * dd.x));
                }
            } else {
                store_split<W>(Sb + (size_t)q * Wp, row, t);
            }
        }
        pend = nobj || chk;
        pchk = chk;
        pnobj = nobj;
        if (!barrier()) {
            alive = false;
            break;
        }
    }
    // the last iteration's decision, if the loop has ended at its limit
    if (alive && pend && k >= kend && service) stop = decide(k, pchk, pnobj);
    // state of iteration k for the next launch, the final transform and the read-out calls
    if (k > k0) {
        float2* __restrict__ d2out = reinterpret_cast<float2*>(P.d2 + (k & 1) * P.d2_stride);
        if (owned) {
#pragma unroll
            for (int m = 0; m < 8; ++m) {
                const size_t pix = (size_t)q * W + t + m * FT;
                d2out[pix] = make_float2(dh[m], dv[m]);
                P.d1[pix] = d1[m];
                P.xprev[pix] = xp_s[(i - 1) * W + t + m * FT];
            }
        }
        if constexpr (DSM) {
            for (int e = tid; e < R * Wc; e += C::NT) Sa[(size_t)(r0 + e / Wc) * Wp + e % Wc] = spec[Wc + e];
            for (int e = tid; e < H * ncol; e += C::NT)
                Sb[(size_t)(e / ncol) * Wp + c0 + e % ncol] = tile[e / ncol * NC + e % ncol];
        }
    }
    if (!alive && tid == 0) atomicExch(&ctl->status, kStatusTimeout);
    if (rank == 0 && service && lane == 0) {
        ctl->team_base = target;
        ctl->iter = k;
        // (0 to this decision's: a wait that ran out in another CTA, at the last barrier alone too, stays)
        if (status != 0) atomicCAS(&ctl->status, 0, status);
        ctl->have_obj = have_obj;
        ctl->obj = obj;
        ctl->obj_prev = obj_prev;
        ctl->rel_x = rel_x;
        ctl->rel_obj = rel_obj;
        ctl->primal_res = primal_res;
        if (conv) ctl->converged = 1;
        if (stop || !alive || k >= max_iters) {
            ctl->active = 0;
            ctl->t_done = device_clock_ns();
            atomicSub(n_active, 1);
        }
    }
}

// The problems of a class of this size in flight at once; 0 if the size has no
// team kernel or the device cannot hold a team
int tv_team_capacity(int H, int W, bool aniso);
bool tv_team_cluster(int H, int W);   // its teams are clusters
cudaError_t launch_tv_team(int H, int W, bool aniso, const ProbDesc* d, SlotTable sl, int slots, int Wp,
                           const float2* tw, int* n_active, int max_steps, cudaStream_t s);

}  // namespace admm
