// gfft.cuh -- shared-memory Stockham FFTs of mixed radix for the lengths
// N = m 2^k, m in {1, 3, 5}, that the exact (unpadded) domains use.
//
// The x-update of the ADMM is diagonal in the DFT domain for any domain size
// (Sec. IV-A: the domain only has to hold the image and the kernel support);
// the power-of-two kernels (fft.cuh) serve sides 64..2048, these serve the
// others (192, 384, 768, 1536; 320, 640, 1280) and, in a domain with one
// such side, the power-of-two side too.
//
// Layout: one length-N transform is owned by a group of T = N / E threads;
// thread t holds, in registers, the E elements t + e T, e = 0..E-1, before
// and after the transform (natural order). E is 8 (m = 1), 12 (m = 3) or 20
// (m = 5). Passes: radix E first (no twiddles; as a 4 x m transform by the
// prime factor algorithm of Good and Thomas, whose index maps need no twiddles
// inside either), then radix 4 as long as possible, then one radix 2 if needed;
// every radix divides E, so each thread takes whole butterflies. Lengths with
// m = 1 run the radix-8 transforms of fft.cuh, which have the same layout.
// Between passes the values go through a shared buffer of N float2 per group at
// swizzled positions (gswz); after the last pass they are in natural order in
// registers already.
//
// Stockham pass of radix r with Ns = product of the earlier radices:
// butterfly j in [0, N / r) takes x[j + q N / r], q = 0..r-1, k = j mod Ns,
// multiplies input q by exp(DIR 2 pi i q k / (r Ns)), applies the r-point DFT
// and writes output q to position (j - k) r + k + q Ns.
//
// DIR = -1: X[k] = sum_n x[n] exp(-2 pi i k n / N) (unnormalised forward)
// DIR = +1: x[n] = sum_k X[k] exp(+2 pi i k n / N) (unnormalised inverse)
//
// Twiddles: per pass one block of (r - 1) Ns entries, (q - 1) Ns + k holding
// exp(-2 pi i q k / (r Ns)), so that the lanes of a warp (consecutive k) read
// consecutive entries; computed in FP64 on the host (fill_gen_table) and staged
// in shared memory by the kernels.
// 8 x 384^2 per launch, against passes of radix 3, 4, 4, 4, 2 with an exchange
// after each and one twiddle table for all: column phase 31.4 -> 21.9 us,
// inverse rows 16.5 -> 12.4, forward rows 13.4 -> 9.4.
#pragma once
#include <cuda_runtime.h>

#include <cmath>

#include "kernels.cuh"

namespace admm {

__host__ __device__ constexpr int gfft_odd(int n) { return (n & 1) ? n : gfft_odd(n >> 1); }
__host__ __device__ constexpr int gfft_log2(int n) { return n <= 1 ? 0 : 1 + gfft_log2(n >> 1); }

// lengths the generic kernels take: m 2^k with m in {1, 3, 5}, a multiple of
// 32 (the tile kernels' tile) and of 16 E / 8 threads' worth, within 64..2048
__host__ __device__ constexpr bool gfft_length_ok(int n) {
    return n >= 64 && n <= 2048 && n % 32 == 0 &&
           (gfft_odd(n) == 1 || gfft_odd(n) == 3 || gfft_odd(n) == 5) &&
           (n / gfft_odd(n)) >= 32;
}

template <int N> struct GShape {
    static_assert(gfft_length_ok(N), "unsupported generic FFT length");
    static constexpr int M = gfft_odd(N);                 // odd factor
    static constexpr int P2 = N / M;                      // power-of-two factor
    static constexpr int E = M == 1 ? 8 : (M == 3 ? 12 : 20);   // elements per thread
    static constexpr int T = N / E;                       // threads per transform
    static constexpr int L2 = gfft_log2(P2) - 2;          // (M > 1: after the leading radix 4 M)
    static constexpr int NPASS = 1 + (L2 + 1) / 2;
    static_assert(T >= 8 && (T <= 32 || T % 32 == 0), "group size");
    __host__ __device__ static constexpr int radix(int p) { return p == 0 ? E : (p - 1 < L2 / 2 ? 4 : 2); }
};

// Host: the per-pass twiddle table of length n = m 2^k, m in {3, 5}, into dst
// (at most n entries); exact reduction of the angles
inline void fill_gen_table(int n, float2* dst) {
    const int m = gfft_odd(n), e = 4 * m;
    int ns = e, o = 0;
    while (ns < n) {
        const int r = n / ns >= 4 ? 4 : 2;
        for (int q = 1; q < r; ++q)
            for (int k = 0; k < ns; ++k) {
                const double a = 2.0 * 3.14159265358979323846 * (double)((long long)q * k) / ((double)r * ns);
                dst[o + (q - 1) * ns + k] = make_float2((float)cos(a), (float)(-sin(a)));
            }
        o += (r - 1) * ns;
        ns *= r;
    }
}

// Swizzled position of element i of an exchange buffer: the low four index bits
// by the next four (a bijection of every 16 elements), which spreads the
// stride-12 and stride-20 stores of the first pass over the banks.
__host__ __device__ constexpr int gswz(int i) { return i ^ ((i >> 4) & 15); }

// r-point DFTs in registers (natural order in and out)
template <int DIR> __device__ __forceinline__ void gdft3(float2& a, float2& b, float2& c) {
    // w = exp(DIR 2 pi i / 3) = -1/2 + DIR i sqrt(3)/2
    const float s = 0.86602540378443864676f;
    const float2 sbc = b + c, dbc = b - c;
    const float2 m = make_float2(a.x - 0.5f * sbc.x, a.y - 0.5f * sbc.y);
    const float2 r = mul_i<DIR>(s * dbc);
    a = a + sbc;
    b = m + r;
    c = m - r;
}

template <int DIR> __device__ __forceinline__ void gdft5(float2& x0, float2& x1, float2& x2, float2& x3, float2& x4) {
    // w = exp(DIR 2 pi i / 5): cos and sin of 2 pi / 5 and 4 pi / 5
    const float c1 = 0.30901699437494742410f, c2 = -0.80901699437494742410f;
    const float s1 = 0.95105651629515357212f, s2 = 0.58778525229247312917f;
    const float2 t1 = x1 + x4, t2 = x2 + x3, t3 = x1 - x4, t4 = x2 - x3;
    const float2 a1 = make_float2(x0.x + c1 * t1.x + c2 * t2.x, x0.y + c1 * t1.y + c2 * t2.y);
    const float2 a2 = make_float2(x0.x + c2 * t1.x + c1 * t2.x, x0.y + c2 * t1.y + c1 * t2.y);
    const float2 b1 = mul_i<DIR>(make_float2(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y));
    const float2 b2 = mul_i<DIR>(make_float2(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y));
    x0 = x0 + t1 + t2;
    x1 = a1 + b1;
    x4 = a1 - b1;
    x2 = a2 + b2;
    x3 = a2 - b2;
}

// barrier over the T threads of transform group g (T <= 32: the group's
// lanes of one warp; else named barrier 1 + g)
template <int T> __device__ __forceinline__ void ggroup_sync(int g) {
    if constexpr (T <= 32) {
        constexpr unsigned lanes = T == 32 ? 0xffffffffu : ((1u << T) - 1u);
        __syncwarp(lanes << ((g * T) & 31));
    } else {
        asm volatile("bar.sync %0, %1;\n" ::"r"(1 + g), "n"(T) : "memory");
    }
}

// E-point DFT of x, E = 4 M, by the prime factor algorithm: input index (M n1 +
// 4 n2) mod E for row n1 < 4, column n2 < M; output index = k1 mod 4, k2 mod M
template <int M, int DIR> __device__ __forceinline__ void gdft_pfa(float2 (&x)[4 * M]) {
    constexpr int E = 4 * M, C2 = M == 3 ? 4 : 16, C1 = M == 3 ? 9 : 5;   // CRT: C1 = 1 mod 4, 0 mod M; C2 the other way
    float2 y[4][M];
#pragma unroll
    for (int n2 = 0; n2 < M; ++n2) {
        float2 a[4];
#pragma unroll
        for (int n1 = 0; n1 < 4; ++n1) a[n1] = x[(M * n1 + 4 * n2) % E];
        // (over n1 the kernel is exp(DIR 2 pi i M n1 k / E) = exp(DIR 2 pi i n1 k / 4))
        dft4<DIR>(a[0], a[1], a[2], a[3]);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) y[k1][n2] = a[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        if constexpr (M == 3) gdft3<DIR>(y[k1][0], y[k1][1], y[k1][2]);
        else gdft5<DIR>(y[k1][0], y[k1][1], y[k1][2], y[k1][3], y[k1][4]);
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) x[(C1 * k1 + C2 * k2) % E] = y[k1][k2];
    }
}

// Transforms of S signals (S buffers of N float2, one after the other from buf)
// on one group: twiddles, index arithmetic and barriers are shared.
//   v   : in/out, element t + e T of signal i in v[i][e] (natural order both ways)
//   tw  : the length's per-pass table (fill_gen_table; m = 1: load_twiddles), shared memory
// The leading barrier orders any earlier reads of buf by the group; after the
// last read of buf the group is synchronised again.
template <int N, int DIR, int S>
__device__ __forceinline__ void gfft_signals(float2 (&v)[S][GShape<N>::E], int t, int g, const float2* tw,
                                             float2* buf) {
    using G = GShape<N>;
    constexpr int E = G::E, T = G::T;
    if constexpr (G::M == 1) {
        if constexpr (S == 2) fft_group2<N, DIR>(v[0], v[1], buf, buf + N, tw, t, g);
        else fft_group<N, DIR>(v[0], buf, tw, t, g);
    } else {
#pragma unroll
        for (int i = 0; i < S; ++i) gdft_pfa<G::M, DIR>(v[i]);
        ggroup_sync<T>(g);
#pragma unroll
        for (int i = 0; i < S; ++i)
#pragma unroll
            for (int e = 0; e < E; ++e) buf[i * N + gswz(E * t + e)] = v[i][e];
        int Ns = E, o = 0;
#pragma unroll
        for (int p = 1; p < G::NPASS; ++p) {
            ggroup_sync<T>(g);
#pragma unroll
            for (int i = 0; i < S; ++i)
#pragma unroll
                for (int e = 0; e < E; ++e) v[i][e] = buf[i * N + gswz(t + T * e)];
            ggroup_sync<T>(g);       // buf may be written again
            const bool four = G::radix(p) == 4, last = p + 1 == G::NPASS;
            const int R = four ? 4 : 2, B = E / R;
#pragma unroll
            for (int b = 0; b < E / 2; ++b) {
                if (b >= B) continue;
                const int j = t + T * b, k = j % Ns;
                const int base = (j - k) * R + k;
                if (four) {
                    const float2 w1 = twid<DIR>(tw + o, k), w2 = twid<DIR>(tw + o, Ns + k), w3 = twid<DIR>(tw + o, 2 * Ns + k);
#pragma unroll
                    for (int i = 0; i < S; ++i) {
                        float2& x0 = v[i][b];
                        float2& x1 = v[i][b + E / 4];
                        float2& x2 = v[i][b + 2 * (E / 4)];
                        float2& x3 = v[i][b + 3 * (E / 4)];
                        x1 = cmul(x1, w1);
                        x2 = cmul(x2, w2);
                        x3 = cmul(x3, w3);
                        dft4<DIR>(x0, x1, x2, x3);
                        if (!last) {
                            buf[i * N + gswz(base)] = x0;
                            buf[i * N + gswz(base + Ns)] = x1;
                            buf[i * N + gswz(base + 2 * Ns)] = x2;
                            buf[i * N + gswz(base + 3 * Ns)] = x3;
                        }
                    }
                } else {
                    const float2 w1 = twid<DIR>(tw + o, k);
#pragma unroll
                    for (int i = 0; i < S; ++i) {
                        float2& x0 = v[i][b];
                        float2& x1 = v[i][b + E / 2];
                        x1 = cmul(x1, w1);
                        dft2<DIR>(x0, x1);
                        if (!last) {
                            buf[i * N + gswz(base)] = x0;
                            buf[i * N + gswz(base + Ns)] = x1;
                        }
                    }
                }
            }
            o += (R - 1) * Ns;
            Ns *= R;
        }
    }
}

// the per-pass table of length N into shared memory (tw_g: the device table of
// this length; m = 1: the 2048-entry table)
template <int N>
__device__ __forceinline__ void load_gen_twiddles(float2* dst, const float2* __restrict__ tw_g, int tid, int nthr) {
    if constexpr (GShape<N>::M == 1) {
        load_twiddles<N>(dst, tw_g, tid, nthr);
    } else {
        for (int e = tid; e < N / 2; e += nthr) cp_async16(dst + 2 * e, tw_g + 2 * e);
        cp_async_commit();
    }
}

}  // namespace admm
