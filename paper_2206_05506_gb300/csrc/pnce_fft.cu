// Correlation with a real-valued pilot by FFT, FP32 on the CUDA cores: the relaxed pilot's
// forward, the received-block half of its adjoint and the pilot half.
//
// With S >= N + K*L - 1 a power of two and q the pilot continued over the indices that occur,
// q[m] = p[m mod N] for -(KL - 1) <= m < N (taken mod S, zero elsewhere),
//     H[j]  = (1/N) sum_n Y[n] q[n - j],  j < KL        IFFT(FFT(Y) conj(FFT(q)))
//     dY[n] = (1/N) sum_j G[j] q[n - j],  n < N         IFFT(FFT(G) FFT(q))
//     r[m]  = sum_a sum_j conj(G[j]) Y[m + j]           IFFT(sum_a conj(FFT(G)) FFT(Y))
//     dp[i] = (1/N) Re(r[i] + r[i - N])
// No index wraps onto another one, so these are the sums of pnce_simt.cu and pnce_adjoint.cu
// in O(log S) operations per sample instead of K*L.
//
// Layout: S = 16 M, one team of M threads per row, 16 values per thread.  M = 16 M2 (M2 <= 16):
// a radix-16 pass over n = n1 M + t, twiddles, an exchange through shared memory, a radix-16
// pass over the M-point parts, twiddles, an exchange within M2 neighbouring lanes, a radix-M2
// pass; the inverse runs the same way back, so no reordering is needed and rows are read and
// written in order straight from and to memory.  The twiddles of a thread (30 values) stay
// in its registers over all its rows, the pilot's spectrum in shared memory.
//
// Bound by instruction issue (about 870 per thread and transform of 2048 points, radix 16, 8
// in the last pass; issue slots 53 % used at 16 warps per SM when a first version was
// profiled), not by memory: 4096 rows of N = 1023, 512 lags move 50 MB.  Against the dense
// sums, same shape: forward 150 -> 42 us, dY 151 -> 44, pilot gradient 180 -> 37 (both together
// share the transform of G); 2048 rows of N = 2047, 300 lags: 189 -> 46, 116 -> 48, 137 -> 43
// us; even with 1-8 lags, where the dense kernel still pays for a tile of 256, N = 1023: 97 ->
// 42 us.  Error against 64 bits, N = 1023: 5e-7 -> 2e-7 (fewer roundings per output).  Lengths
// above 4096 (N + K*L - 1) stay with the dense kernels, and so do the shapes where these are the
// more exact ones (fft_forward_applies, fft_adjoint_applies).
//
// A row whose values are not numbers, or so large that an intermediate overflows, comes out
// of the transforms as infinities and NaN throughout; every such output is summed again
// directly, in the order of the dense kernel (the pilot gradient: direct_dp).
#include <algorithm>

#include "pnce_internal.h"

namespace {

constexpr int MIN_LOG = 7, MAX_LOG = 12;       // transform lengths 128 .. 4096
constexpr int MIN_ADJOINT_LOG = 8;             // of the adjoint (128 lags and more)

template <int LS>
struct Fft {
    static constexpr int S = 1 << LS, M = S / 16;
    static constexpr int M2 = M >= 16 ? M / 16 : 1;           // length of the third pass
    static constexpr bool TWO = M < 16;                      // two passes: 16 and M
    static constexpr int R = TWO ? M : M2;                   // length of the last pass
    static constexpr int GR = 16 / R;                        // its groups per thread
    static constexpr int THREADS = M < 128 ? (M == 64 ? 64 : 128) : M;
    static constexpr int RT = THREADS / M;                   // rows per block
    static constexpr int LD1 = M + (TWO ? 1 : M2 < 16 ? M2 : 0);
    static constexpr int X1 = 16 * LD1;                      // first exchange, entries
    static constexpr int LD2 = 16 * (M2 + 1) + M2;
    static constexpr int X2 = M2 > 1 ? 16 * LD2 : 0;         // second exchange, same buffer
    // direct_sums: one entry of padding per 16, and 16 outputs past the last one
    static constexpr int XD = S + S / 16 + 32;
    static constexpr int ROW = std::max(std::max(X1, X2), XD);
    static constexpr int TW2 = M2 > 1 ? 15 * M2 : 0;         // second twiddles, [k - 1][m2]
    // entries of dynamic shared memory: a spectrum, the second twiddles, the rows' buffers
    static constexpr int SMEM = S + (TW2 + 1) / 2 * 2 + RT * ROW;
    // blocks per SM, by registers: about 100 a thread forward, 120 for dY alone, 170 with the
    // pilot gradient
    static constexpr int BPS = THREADS == 256 ? 2 : THREADS == 64 ? 8 : 5;
    static constexpr int DY_BPS = THREADS == 256 ? 2 : THREADS == 64 ? 8 : 4;
    static constexpr int DP_BPS = THREADS == 256 ? 1 : THREADS == 64 ? 5 : 3;
};

template <int M>
__device__ __forceinline__ void row_sync() {
    if constexpr (M <= 32)
        __syncwarp();
    else
        __syncthreads();
}

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
// a w, or a conj(w)
template <bool CONJ>
__device__ __forceinline__ float2 cmul(float2 a, float2 w) {
    const float s = CONJ ? -w.y : w.y;
    return make_float2(fmaf(a.x, w.x, -a.y * s), fmaf(a.x, s, a.y * w.x));
}

// whether bad is true in any of the row's threads (M <= 32: of its warp's)
template <int M>
__device__ __forceinline__ bool row_any(bool bad) {
    if constexpr (M <= 32)
        return __any_sync(0xffffffffu, bad);
    else
        return __syncthreads_or(bad);
}

// DFT of length 2, 4, 8, 16 on v[B], v[B + D], ..; results in order.  INV: exponent +.
template <bool INV, int E>
__device__ __forceinline__ void dft4(float2 (&v)[E], int i0, int i1, int i2, int i3) {
    const float2 s0 = cadd(v[i0], v[i2]), s1 = csub(v[i0], v[i2]);
    const float2 s2 = cadd(v[i1], v[i3]), d = csub(v[i1], v[i3]);
    v[i0] = cadd(s0, s2);
    v[i2] = csub(s0, s2);
    const float2 up = make_float2(s1.x - d.y, s1.y + d.x);       // s1 + i d
    const float2 dn = make_float2(s1.x + d.y, s1.y - d.x);       // s1 - i d
    v[i1] = INV ? up : dn;
    v[i3] = INV ? dn : up;
}

// the same with v[i2] = v[i3] = 0
template <bool INV, int E>
__device__ __forceinline__ void dft4_half(float2 (&v)[E], int i0, int i1, int i2, int i3) {
    const float2 a = v[i0], b = v[i1];
    const float2 up = make_float2(a.x - b.y, a.y + b.x), dn = make_float2(a.x + b.y, a.y - b.x);
    v[i0] = cadd(a, b);
    v[i2] = csub(a, b);
    v[i1] = INV ? up : dn;
    v[i3] = INV ? dn : up;
}

// HALF: the inputs v[8 ..] are zero (and need not be set)
template <bool INV, bool HALF = false>
__device__ __forceinline__ void dft16(float2 (&v)[16]) {
    // n = 4 a + b: DFT4 over a for every b, twiddles W16^(b k), DFT4 over b
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        if constexpr (HALF)
            dft4_half<INV>(v, b, 4 + b, 8 + b, 12 + b);
        else
            dft4<INV>(v, b, 4 + b, 8 + b, 12 + b);
    }
    constexpr float C1 = 0.92387953251128675613f, S1 = 0.38268343236508977173f,
                    H = 0.70710678118654752440f;
    const float2 w1 = make_float2(C1, -S1), w2 = make_float2(H, -H), w3 = make_float2(S1, -C1);
    // v[4 k + b] times W16^(k b)
    v[4 + 1] = cmul<INV>(v[4 + 1], w1);
    v[4 + 2] = cmul<INV>(v[4 + 2], w2);
    v[4 + 3] = cmul<INV>(v[4 + 3], w3);
    v[8 + 1] = cmul<INV>(v[8 + 1], w2);
    v[8 + 2] = INV ? make_float2(-v[8 + 2].y, v[8 + 2].x) : make_float2(v[8 + 2].y, -v[8 + 2].x);
    v[8 + 3] = cmul<INV>(v[8 + 3], make_float2(-H, -H));
    v[12 + 1] = cmul<INV>(v[12 + 1], w3);
    v[12 + 2] = cmul<INV>(v[12 + 2], make_float2(-H, -H));
    v[12 + 3] = cmul<INV>(v[12 + 3], make_float2(-C1, S1));
#pragma unroll
    for (int k = 0; k < 4; ++k) dft4<INV>(v, 4 * k, 4 * k + 1, 4 * k + 2, 4 * k + 3);
    // v[4 k1 + k2] holds X[k1 + 4 k2]
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
        for (int k2 = k1 + 1; k2 < 4; ++k2) {
            const float2 t = v[4 * k1 + k2];
            v[4 * k1 + k2] = v[4 * k2 + k1];
            v[4 * k2 + k1] = t;
        }
}

// 16 / R DFTs of length R, group g on v[g R .. g R + R)
template <bool INV, int R>
__device__ __forceinline__ void dft_groups(float2 (&v)[16]) {
    if constexpr (R == 16) {
        dft16<INV>(v);
    } else if constexpr (R == 8) {
        constexpr float H = 0.70710678118654752440f;
#pragma unroll
        for (int g = 0; g < 16; g += 8) {
            float2 e[4] = {v[g], v[g + 2], v[g + 4], v[g + 6]};
            float2 o[4] = {v[g + 1], v[g + 3], v[g + 5], v[g + 7]};
            dft4<INV>(e, 0, 1, 2, 3);
            dft4<INV>(o, 0, 1, 2, 3);
            o[1] = cmul<INV>(o[1], make_float2(H, -H));
            o[2] = INV ? make_float2(-o[2].y, o[2].x) : make_float2(o[2].y, -o[2].x);
            o[3] = cmul<INV>(o[3], make_float2(-H, -H));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v[g + k] = cadd(e[k], o[k]);
                v[g + 4 + k] = csub(e[k], o[k]);
            }
        }
    } else if constexpr (R == 4) {
#pragma unroll
        for (int g = 0; g < 16; g += 4) dft4<INV>(v, g, g + 1, g + 2, g + 3);
    } else if constexpr (R == 2) {
#pragma unroll
        for (int g = 0; g < 16; g += 2) {
            const float2 a = v[g], b = v[g + 1];
            v[g] = cadd(a, b);
            v[g + 1] = csub(a, b);
        }
    }
}

// exp(-2 pi i k / n)
__device__ __forceinline__ float2 root(int k, int n) {
    float s, c;
    sincospif(-2.0f * (float)k / (float)n, &s, &c);    // k < n <= 4096: the quotient is exact
    return make_float2(c, s);
}

// W_M^(m2 k) for the block, [k - 1][m2]
template <int LS>
__device__ __forceinline__ void fill_tw2(float2* tw2) {
    using F = Fft<LS>;
    for (int i = threadIdx.x; i < F::TW2; i += F::THREADS)
        tw2[i] = root((i % F::M2) * (i / F::M2 + 1) & (F::M - 1), F::M);
}

template <int LS>
struct Team {
    using F = Fft<LS>;
    float2* x;           // this row's exchange buffer
    const float2* tw2;   // the block's second twiddles
    int t;               // thread of the row's team: n2 of the first pass, (f1, m2) of the second
    float2 tw1[15];      // W_S^(t k), k = 1 .. 15

    __device__ __forceinline__ Team(float2* buf, const float2* tw, int t_) : x(buf), tw2(tw), t(t_) {
#pragma unroll
        for (int k = 1; k < 16; ++k) tw1[k - 1] = root(t * k & (F::S - 1), F::S);
    }

    // v[n1] = x[n1 M + t] -> the row's spectrum in the team's own order.  HALF: v[8 ..] = 0
    template <bool HALF>
    __device__ __forceinline__ void forward(float2 (&v)[16]) {
        dft16<false, HALF>(v);
#pragma unroll
        for (int k = 1; k < 16; ++k) v[k] = cmul<false>(v[k], tw1[k - 1]);
        row_sync<F::M>();                          // the buffer's last readers are done
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k * F::LD1 + t] = v[k];
        row_sync<F::M>();
        if constexpr (F::TWO) {
#pragma unroll
            for (int g = 0; g < F::GR; ++g)
#pragma unroll
                for (int m = 0; m < F::M; ++m)
                    v[g * F::M + m] = x[(t + F::M * g) * F::LD1 + m];
            dft_groups<false, F::M>(v);
        } else {
            const int f1 = t / F::M2, m2 = t % F::M2;
#pragma unroll
            for (int m = 0; m < 16; ++m) v[m] = x[f1 * F::LD1 + m * F::M2 + m2];
            dft16<false>(v);
            if constexpr (F::M2 > 1) {
#pragma unroll
                for (int k = 1; k < 16; ++k) v[k] = cmul<false>(v[k], tw2[(k - 1) * F::M2 + m2]);
                float2* b = x + f1 * F::LD2;
                row_sync<F::M>();                  // the first exchange is read
#pragma unroll
                for (int k = 0; k < 16; ++k) b[k * (F::M2 + 1) + m2] = v[k];
                __syncwarp();                      // M2 neighbouring lanes exchange
#pragma unroll
                for (int g = 0; g < F::GR; ++g)
#pragma unroll
                    for (int m = 0; m < F::M2; ++m)
                        v[g * F::M2 + m] = b[(m2 + F::M2 * g) * (F::M2 + 1) + m];
                dft_groups<false, F::M2>(v);
            }
        }
    }

    // the way back; v[n1] = S x[n1 M + t]
    __device__ __forceinline__ void inverse(float2 (&v)[16]) {
        if constexpr (F::TWO) {
            dft_groups<true, F::M>(v);
            row_sync<F::M>();
#pragma unroll
            for (int g = 0; g < F::GR; ++g)
#pragma unroll
                for (int m = 0; m < F::M; ++m)
                    x[(t + F::M * g) * F::LD1 + m] = v[g * F::M + m];
        } else {
            const int f1 = t / F::M2, m2 = t % F::M2;
            if constexpr (F::M2 > 1) {
                dft_groups<true, F::M2>(v);
                float2* b = x + f1 * F::LD2;
                __syncwarp();                      // only these lanes use this part since
#pragma unroll
                for (int g = 0; g < F::GR; ++g)
#pragma unroll
                    for (int m = 0; m < F::M2; ++m)
                        b[(m2 + F::M2 * g) * (F::M2 + 1) + m] = v[g * F::M2 + m];
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = b[k * (F::M2 + 1) + m2];
#pragma unroll
                for (int k = 1; k < 16; ++k) v[k] = cmul<true>(v[k], tw2[(k - 1) * F::M2 + m2]);
            }
            dft16<true>(v);
            row_sync<F::M>();
#pragma unroll
            for (int m = 0; m < 16; ++m) x[f1 * F::LD1 + m * F::M2 + m2] = v[m];
        }
        row_sync<F::M>();
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = x[k * F::LD1 + t];
#pragma unroll
        for (int k = 1; k < 16; ++k) v[k] = cmul<true>(v[k], tw1[k - 1]);
        dft16<true>(v);
    }
};

// row[n] for n = k M + t < len, zero from there on (HALF: len <= S / 2, v[8 ..] is not set)
template <int LS, bool HALF>
__device__ __forceinline__ void load_row(float2 (&v)[16], const float2* row, int len, int t) {
#pragma unroll
    for (int k = 0; k < (HALF ? 8 : 16); ++k) {
        const int n = k * Fft<LS>::M + t;
        v[k] = n < len ? __ldg(row + n) : make_float2(0.f, 0.f);
    }
}

__device__ __forceinline__ float pilot_at(const float* p, bool tanh_map, int i) {
    const float v = __ldg(p + i);
    return tanh_map ? tanhf(v) : v;
}

// The pilot's spectrum of the block, [k][t]; ends with the block synchronised.
template <int LS>
__device__ __forceinline__ void pilot_spectrum(Team<LS>& team, const float* p, bool tanh_map, int N,
                                               int KL, int sub, float2* Q) {
    using F = Fft<LS>;
    float2 v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int m = k * F::M + team.t;
        const int i = m < N ? m : m > F::S - KL ? N + m - F::S : -1;
        v[k] = make_float2(i >= 0 ? pilot_at(p, tanh_map, i) : 0.f, 0.f);
    }
    team.template forward<false>(v);       // every row of the block; the first one keeps it
    if (sub == 0) {
#pragma unroll
        for (int k = 0; k < 16; ++k) Q[k * F::M + team.t] = v[k];
    }
    __syncthreads();
}

// acc[r] += in[k] e[16 t + r + k] for k = 0, 1, .. in order (real parts and imaginary parts apart),
// with e[q] at x[q + q / 16]: 16 consecutive outputs per thread, so that a step of one k takes one
// new entry of e, its 8-byte loads free of bank conflicts.
__device__ __forceinline__ void direct_sums(float2 (&acc)[16], const float2* x, const float2* in,
                                            int in_len, int t) {
    const float2* e = x + 17 * t;
    float2 w[31];
#pragma unroll
    for (int i = 0; i < 15; ++i) w[i] = e[i];
    int k = 0;
#pragma unroll 1
    for (; k + 16 <= in_len; k += 16, e += 17, in += 16) {
        w[15] = e[15];
#pragma unroll
        for (int i = 16; i < 31; ++i) w[i] = e[i + 1];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            const float2 v = __ldg(in + u);
#pragma unroll
            for (int r = 0; r < 16; ++r) acc[r] = __ffma2_rn(v, w[r + u], acc[r]);
        }
#pragma unroll
        for (int i = 0; i < 15; ++i) w[i] = w[i + 16];
    }
    for (int u = 0; k < in_len; ++k, ++u) {
        const float2 v = __ldg(in + u);
#pragma unroll
        for (int r = 0; r < 16; ++r) acc[r] = __ffma2_rn(v, e[r + u + (r + u) / 16], acc[r]);
    }
}

// The block's rows once more, after it has stored them all: out[o] = (1/N) sum_{k < in_len} in[k]
// pilot[(k - o) mod N] (ADJ: pilot[(o - k) mod N]) for the outputs that are not finite, the products
// summed in order as the dense kernel does.  Behind the loop over the rows, so that it costs that
// loop no registers and no barrier.  4096 rows of N = 1023, 512 lags, a NaN in every row, us:
// forward 352 (43 without; the dense kernel 152), dY 272 (45; 154); one output per thread and pass,
// as it was before, 2530 and 2984.
template <int LS, bool ADJ>
__device__ __noinline__ void direct_rows(float2* x, const float2* in, int in_len, float2* out,
                                         int out_len, long long A, const float* p, bool tanh_map,
                                         int N, int sub, int t) {
    using F = Fft<LS>;
    const float invN = 1.0f / (float)N;
    for (long long first = (long long)blockIdx.x * F::RT; first < A;
         first += (long long)gridDim.x * F::RT) {
        const bool live = first + sub < A;
        const long long row = live ? first + sub : first;
        float2* const o_row = out + row * out_len;
        bool bad = false;
        for (int o = t; live && o < out_len; o += F::M)
            bad |= !(isfinite(o_row[o].x) && isfinite(o_row[o].y));
        if (!row_any<F::M>(bad)) continue;
        // output out_len - 1 - i takes the pilot's sample for k at e[i + k]
        for (int q = t; q < in_len + out_len - 1; q += F::M) {
            const int m = ADJ ? N - 1 - q : q - (out_len - 1);
            const float w = pilot_at(p, tanh_map, m < 0 ? m + N : m);
            x[q + q / 16] = make_float2(w, w);
        }
        row_sync<F::M>();
        if (live && 16 * t < out_len) {
            float2 acc[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) acc[r] = make_float2(0.f, 0.f);
            direct_sums(acc, x, in + row * in_len, in_len, t);
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int o = out_len - 1 - 16 * t - r;
                if (o >= 0 && !(isfinite(o_row[o].x) && isfinite(o_row[o].y)))
                    o_row[o] = make_float2(acc[r].x * invN, acc[r].y * invN);
            }
        }
        row_sync<F::M>();
    }
}

// out[o] = v scale for o < out_len; whether all of them are finite
template <int LS>
__device__ __forceinline__ bool store_row(float2 (&v)[16], float2* out, int out_len, int t, int N) {
    using F = Fft<LS>;
    const float scale = 1.0f / ((float)N * (float)F::S);
    bool fine = true;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const int o = k * F::M + t;
        if (o < out_len) {
            const float2 w = make_float2(v[k].x * scale, v[k].y * scale);
            // 0 x is 0 for finite x, NaN otherwise
            fine = fine && fmaf(0.f, w.x, 0.f * w.y) == 0.f;
            out[o] = w;
        }
    }
    return fine;
}

// Forward: A rows Y of N samples -> KL lags.  HALF: N <= S / 2.
template <int LS, bool HALF>
__global__ void __launch_bounds__(Fft<LS>::THREADS, Fft<LS>::BPS)
fft_forward_kernel(const float* __restrict__ p, bool tanh_map, const float2* __restrict__ Y,
                   long long A, int N, int KL, float2* __restrict__ H) {
    using F = Fft<LS>;
    extern __shared__ __align__(16) float2 fft_smem[];
    float2 *Q = fft_smem, *tw2 = Q + F::S;
    const int sub = threadIdx.x / F::M, t = threadIdx.x % F::M;
    fill_tw2<LS>(tw2);
    Team<LS> team(fft_smem + F::SMEM - (F::RT - sub) * F::ROW, tw2, t);
    __syncthreads();
    pilot_spectrum<LS>(team, p, tanh_map, N, KL, sub, Q);
    bool fine = true;
    for (long long r0 = (long long)blockIdx.x * F::RT; r0 < A; r0 += (long long)gridDim.x * F::RT) {
        const long long row = r0 + sub;
        const bool live = row < A;
        float2 v[16];
        load_row<LS, HALF>(v, Y + row * N, live ? N : 0, t);
        team.template forward<HALF>(v);
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = cmul<true>(v[k], Q[k * F::M + t]);
        team.inverse(v);
        fine &= store_row<LS>(v, H + row * KL, live ? KL : 0, t, N);
    }
    if (__syncthreads_or(!fine))
        direct_rows<LS, false>(team.x, Y, N, H, KL, A, p, tanh_map, N, sub, t);
}

// The pilot gradient's sums of the rows row0, row0 + stride, .. (row0 = first + sub) formed
// directly, in order: slot[i] = (NaN, r[i] + r[i - N]) for i < N, (NaN, 0) above.  In place of a
// spectrum that is not finite: the NaN marks the slot, and fft_dp_final_kernel adds the sums.  Every block does this
// for its own rows, so that such a row costs its block's rows a direct sum and no more.  Pilot
// gradient of 4096 rows of N = 1023, 512 lags, us: 38.8; a NaN in one row 179, in every row 293 (the
// dense kernel 182; every entry summed by itself in fft_dp_final_kernel: 146000).
template <int LS>
__device__ __noinline__ void direct_dp(const float2* G, const float2* Y, long long first, int sub,
                                       long long stride, long long A, int N, int KL, int t,
                                       float2* x, float2* slot) {
    float2 acc[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) acc[r] = make_float2(0.f, 0.f);
    for (; first < A; first += stride) {
        const long long row = first + sub;
        if (row < A) {
            const float2* y = Y + row * N;
            for (int q = t; q < N + KL - 1; q += Fft<LS>::M) x[q + q / 16] = __ldg(y + (q < N ? q : q - N));
        }
        row_sync<Fft<LS>::M>();
        if (row < A && 16 * t < N) direct_sums(acc, x, G + row * KL, KL, t);
        row_sync<Fft<LS>::M>();
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) slot[16 * t + r] = make_float2(nanf(""), acc[r].x + acc[r].y);
}

// Adjoint.  Block b takes the rows b, b + blocks, .. in order; per row the spectrum of G gives
// dY (times the pilot's) and, times the conjugate, meets that of Y: DP adds these products
// over the block's rows and stores the sum, [k][t].  The number of blocks depends on the
// shape only, so that results do not depend on the device.
template <int LS, bool HALF, bool DY, bool DP>
__global__ void __launch_bounds__(Fft<LS>::THREADS, DP ? Fft<LS>::DP_BPS : Fft<LS>::DY_BPS)
fft_adjoint_kernel(const float* __restrict__ p, bool tanh_map, const float2* __restrict__ G,
                   const float2* __restrict__ Y, long long A, int N, int KL,
                   float2* __restrict__ dY, float2* __restrict__ partial) {
    using F = Fft<LS>;
    extern __shared__ __align__(16) float2 fft_smem[];
    float2 *Q = fft_smem, *tw2 = Q + F::S;
    const int sub = threadIdx.x / F::M, t = threadIdx.x % F::M;
    fill_tw2<LS>(tw2);
    Team<LS> team(fft_smem + F::SMEM - (F::RT - sub) * F::ROW, tw2, t);
    __syncthreads();
    if constexpr (DY) pilot_spectrum<LS>(team, p, tanh_map, N, KL, sub, Q);
    float2 acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = make_float2(0.f, 0.f);
    bool y_fine = true;
    for (long long r0 = (long long)blockIdx.x * F::RT; r0 < A; r0 += (long long)gridDim.x * F::RT) {
        const long long row = r0 + sub;
        const bool live = row < A;
        float2 g[16], v[16];
        load_row<LS, true>(g, G + row * KL, live ? KL : 0, t);     // KL <= N, so KL <= S / 2
        team.template forward<true>(g);
        if constexpr (DY) {
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = cmul<false>(g[k], Q[k * F::M + t]);
            team.inverse(v);
            y_fine &= store_row<LS>(v, dY + row * N, live ? N : 0, t, N);
        }
        if constexpr (DP) {
            load_row<LS, HALF>(v, Y + row * N, live ? N : 0, t);
            team.template forward<HALF>(v);
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                acc[k].x = fmaf(g[k].x, v[k].x, fmaf(g[k].y, v[k].y, acc[k].x));
                acc[k].y = fmaf(g[k].x, v[k].y, fmaf(-g[k].y, v[k].x, acc[k].y));
            }
        }
    }
    if constexpr (DP) {
        float2* o = partial + ((long long)blockIdx.x * F::RT + sub) * F::S;
        bool fine = true;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            fine = fine && fmaf(0.f, acc[k].x, 0.f * acc[k].y) == 0.f;
            o[k * F::M + t] = acc[k];
        }
        if (__syncthreads_or(!fine))
            direct_dp<LS>(G, Y, (long long)blockIdx.x * F::RT, sub, (long long)gridDim.x * F::RT, A,
                          N, KL, t, team.x, o);
    }
    if constexpr (DY) {
        if (__syncthreads_or(!y_fine))
            direct_rows<LS, true>(team.x, G, KL, dY, N, A, p, tanh_map, N, sub, t);
    }
}

// A slot of direct sums (direct_dp) counts as zero among the spectra.
__device__ __forceinline__ float2 spectrum_of(float2 q) {
    return isnan(q.x) ? make_float2(0.f, 0.f) : q;
}

// spec[i] = sum over the P partial spectra, in a fixed order: warp w of a block adds
// w, w + 32, .. for 32 consecutive i, then the 32 sums in order.  *direct: whether slots hold
// direct sums.  A programmatic dependent (partial is not declared restrict: its loads must stay
// behind the wait).
__global__ void __launch_bounds__(1024)
fft_dp_sum_kernel(const float2* partial, int P, int S, float2* spec, int* direct) {
    __shared__ float2 red[32][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float2 s = make_float2(0.f, 0.f);
    bool any = false;
#pragma unroll 8
    for (int b = warp; b < P; b += 32) s = cadd(s, partial[(long long)b * S + i]);
    if (isnan(s.x)) {                          // slots of direct sums: once more without them
        s = make_float2(0.f, 0.f);
        for (int b = warp; b < P; b += 32) {
            const float2 q = partial[(long long)b * S + i];
            any |= isnan(q.x);
            s = cadd(s, spectrum_of(q));
        }
    }
    red[warp][lane] = s;
    any = __syncthreads_or(any);
    if (warp == 0) {
        float2 r = make_float2(0.f, 0.f);
#pragma unroll
        for (int w = 0; w < 32; ++w) r = cadd(r, red[w][lane]);
        spec[i] = r;
        if (i == 0) *direct = any;
    }
}

// Every block: r = IFFT(spec), then for its 32 consecutive i, dp[i] = (1/N) Re(r[i] + r[i - N])
// (times 1 - tanh(theta)^2), plus the direct sums where there are any.  Where that is not finite,
// the sum of the spectra or its transform may have overflowed: the block then adds the spectra
// again scaled by 2^-20 (slots times S is less, so that no sum can overflow) and transforms that.
// A programmatic dependent.
template <int LS>
__global__ void __launch_bounds__(Fft<LS>::THREADS)
fft_dp_final_kernel(const float2* spec, const float2* partial, int P, const int* direct, int N,
                    int KL, const float* __restrict__ theta, float* __restrict__ dp) {
    using F = Fft<LS>;
    extern __shared__ __align__(16) float2 fft_smem[];
    __shared__ float red[F::THREADS];
    float* r = reinterpret_cast<float*>(fft_smem);
    float2* tw2 = fft_smem + F::S;
    const int sub = threadIdx.x / F::M, t = threadIdx.x % F::M;
    fill_tw2<LS>(tw2);
    Team<LS> team(fft_smem + F::SMEM - (F::RT - sub) * F::ROW, tw2, t);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float2 v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = spec[k * F::M + t];
    const bool any = *direct != 0;
    team.inverse(v);
    if (sub == 0) {
#pragma unroll
        for (int k = 0; k < 16; ++k) r[k * F::M + t] = v[k].x;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    if (any) {
        float x = 0.f;
        if (i < N) {
#pragma unroll 4
            for (int b = warp; b < P; b += F::THREADS / 32) {
                const float2 q = partial[(long long)b * F::S + i];
                x += isnan(q.x) ? q.y : 0.f;
            }
        }
        red[threadIdx.x] = x;
    }
    __syncthreads();
    const float scale = 1.0f / ((float)N * (float)F::S);
    float deriv = 1.f, s = 0.f, x = 0.f;
    if (warp == 0 && i < N) {
        if (theta) {
            const float th = tanhf(theta[i]);
            deriv = 1.0f - th * th;
        }
        s = (i > N - KL ? r[i] + r[F::S + i - N] : r[i]) * scale;
        if (any) {
            for (int w = 0; w < F::THREADS / 32; ++w) x += red[32 * w + lane];
            x *= 1.0f / (float)N;
        }
        dp[i] = (s + x) * deriv;
    }
    if (!__syncthreads_or(!isfinite(s))) return;
    const float down = 0x1p-20f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        v[k] = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int b = sub; b < P; b += F::RT)
            v[k] = __ffma2_rn(spectrum_of(partial[(long long)b * F::S + k * F::M + t]),
                              make_float2(down, down), v[k]);
    }
    team.inverse(v);
    for (int w = 0; w < F::RT; ++w) {
        if (sub == w) {
#pragma unroll
            for (int k = 0; k < 16; ++k) r[k * F::M + t] = (w ? r[k * F::M + t] : 0.f) + v[k].x;
        }
        __syncthreads();
    }
    if (warp == 0 && i < N && !isfinite(s)) {
        s = (i > N - KL ? r[i] + r[F::S + i - N] : r[i]) * (scale / down);
        dp[i] = (s + x) * deriv;
    }
}

template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kern)(KArgs...), unsigned grid, unsigned block, size_t smem,
                             cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int LS>
struct Launch {
    using F = Fft<LS>;
    static constexpr size_t smem = sizeof(float2) * F::SMEM;
    using Forward = decltype(&fft_forward_kernel<LS, true>);
    using Adjoint = decltype(&fft_adjoint_kernel<LS, true, true, true>);

    static Forward forward_of(int N) {
        return N <= F::S / 2 ? fft_forward_kernel<LS, true> : fft_forward_kernel<LS, false>;
    }
    static Adjoint adjoint_of(int N, bool dy, bool dp) {
        if (!dp) return fft_adjoint_kernel<LS, true, true, false>;
        if (N <= F::S / 2)
            return dy ? fft_adjoint_kernel<LS, true, true, true>
                      : fft_adjoint_kernel<LS, true, false, true>;
        return dy ? fft_adjoint_kernel<LS, false, true, true>
                  : fft_adjoint_kernel<LS, false, false, true>;
    }
    template <class K>
    static cudaError_t limit(K kern) {
        if (smem <= 48 * 1024) return cudaSuccess;
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    // blocks of the adjoint: one wave on 152 SMs
    static int adjoint_blocks(long long A, bool dp) {
        return (int)std::min<long long>((A + F::RT - 1) / F::RT,
                                        152 * (dp ? F::DP_BPS : F::DY_BPS));
    }

    static cudaError_t forward(const float* p, bool tanh_map, const float2* Y, long long A, int N,
                               int KL, float2* H, cudaStream_t s) {
        auto kern = forward_of(N);
        cudaError_t e = limit(kern);
        if (e != cudaSuccess) return e;
        const unsigned grid =
            (unsigned)std::min<long long>((A + F::RT - 1) / F::RT, 152 * F::BPS);
        kern<<<grid, F::THREADS, smem, s>>>(p, tanh_map, Y, A, N, KL, H);
        return cudaGetLastError();
    }

    static size_t workspace(long long A) {
        // the sum, the partial spectra, fft_dp_sum_kernel's flag
        return sizeof(float2) * ((size_t)F::S * ((size_t)adjoint_blocks(A, true) * F::RT + 1) + 1);
    }

    static cudaError_t adjoint(const float* p, bool tanh_map, const float2* G, const float2* Y,
                               long long A, int N, int KL, float2* dY, float* dp, void* ws,
                               cudaStream_t s) {
        auto kern = adjoint_of(N, dY != nullptr, dp != nullptr);
        cudaError_t e = limit(kern);
        if (e != cudaSuccess) return e;
        float2* spec = static_cast<float2*>(ws);
        const int blocks = adjoint_blocks(A, dp != nullptr);
        kern<<<blocks, F::THREADS, smem, s>>>(p, tanh_map, G, Y, A, N, KL, dY,
                                              dp ? spec + F::S : nullptr);
        if ((e = cudaGetLastError()) != cudaSuccess || !dp) return e;
        const int slots = blocks * F::RT;
        const float2* partial = spec + F::S;
        int* direct = reinterpret_cast<int*>(spec + (size_t)F::S * (slots + 1));
        if ((e = launch_dependent(fft_dp_sum_kernel, F::S / 32, 1024, 0, s, partial, slots, F::S,
                                  spec, direct)) != cudaSuccess)
            return e;
        if ((e = limit(fft_dp_final_kernel<LS>)) != cudaSuccess) return e;
        return launch_dependent(fft_dp_final_kernel<LS>, (unsigned)((N + 31) / 32), F::THREADS, smem,
                                s, (const float2*)spec, partial, slots, (const int*)direct, N, KL,
                                tanh_map ? p : (const float*)nullptr, dp);
    }
};

// Calls f(Launch<LS>) for the transform length of the shape, 2^MIN at least; def where there is
// none.
template <int MIN, class Fn, class T>
T with_length(int N, int KL, T def, Fn f) {
    int ls = MIN;
    while (ls <= MAX_LOG && (1 << ls) < N + KL - 1) ++ls;
    if constexpr (MIN <= 7) {
        if (ls == 7) return f(Launch<7>());
    }
    switch (ls) {
        case 8: return f(Launch<8>());
        case 9: return f(Launch<9>());
        case 10: return f(Launch<10>());
        case 11: return f(Launch<11>());
        case 12: return f(Launch<12>());
        default: return def;
    }
}

}  // namespace

namespace pnce {

static bool fft_applies(int N, int KL) { return N + KL - 1 <= 1 << MAX_LOG; }

// The forward sums N terms, and for short pilots the dense sum of them is the more exact one.
// Error against 64 bits, transform over dense, 400 rows, at the lag count where it is largest: N = 31
// 1.5, N = 62 1.18, N = 64 1.06, N = 71 1.07, N = 83 1.04; N = 84 .. 130 0.77 .. 0.99, N = 2047 0.16.
bool fft_forward_applies(int N, int KL) { return N >= 84 && fft_applies(N, KL); }

// The adjoint sums K*L terms (dY) or rows times K*L of them (pilot gradient): with few lags the
// dense kernels are the more exact ones.  Relative error against 64 bits, dense / transform: dY, 300
// rows, N = 1023, 8 lags 5.9e-8 / 1.5e-7, 64 lags 1.5e-7 / 1.6e-7, 255 lags 2.9e-7 / 1.8e-7; N = 300,
// 75 lags 1.6e-7 / 1.7e-7, 150 lags 2.2e-7 / 1.8e-7; pilot gradient, 40 rows, N = 200, 48 lags
// 1.5e-7 / 2.3e-7, N = 2047, 64 lags 1.7e-7 / 2.0e-7, N = 300, 96 lags 1.9e-7 / 2.1e-7; from 128 lags
// on it is no larger by transform for any of 1 to 2048 rows, N = 128 to 2047.
bool fft_adjoint_applies(int N, int KL) { return KL >= 128 && fft_applies(N, KL); }

cudaError_t launch_fft_forward(const float* p, bool tanh_map, const float2* Y, long long A, int N,
                               int KL, float2* H, cudaStream_t s) {
    if (A <= 0) return cudaSuccess;
    return with_length<MIN_LOG>(N, KL, cudaErrorNotSupported, [&](auto l) {
        return l.forward(p, tanh_map, Y, A, N, KL, H, s);
    });
}

size_t fft_adjoint_workspace(long long A, int N, int KL) {
    return with_length<MIN_ADJOINT_LOG>(N, KL, (size_t)0, [&](auto l) { return l.workspace(A); });
}

cudaError_t launch_fft_adjoint(const float* p, bool tanh_map, const float2* G, const float2* Y,
                               long long A, int N, int KL, float2* dY, float* dp, void* ws,
                               cudaStream_t s) {
    if (A <= 0 || (!dY && !dp)) return cudaSuccess;
    return with_length<MIN_ADJOINT_LOG>(N, KL, cudaErrorNotSupported, [&](auto l) {
        return l.adjoint(p, tanh_map, G, Y, A, N, KL, dY, dp, ws, s);
    });
}

}  // namespace pnce
