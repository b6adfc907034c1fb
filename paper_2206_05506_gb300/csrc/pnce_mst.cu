// Correlation with an m-sequence pilot by the fast m-sequence transform, FP32 on the CUDA
// cores.  For an m-sequence of degree r (N = 2^r - 1) the r-bit windows s_n of the pilot bits
// run through every nonzero vector once and every bit is a GF(2)-linear function of any
// window: p[(n - j) mod N] = (-1)^<u_j, s_n>.  So the correlation of Eq. 3 is
//     N H[j] = W[u_j],   W = Walsh-Hadamard transform of X,  X[s_n] = y[n], X[0] = 0
// (tables s_n and u_j: pnce_fmt_tables): r levels of additions per row instead of K*L
// multiply-adds per sample, each output still a sum of +-y.
//
// What bounds it: HBM (8 bytes a sample in, 8 a lag out), provided that the shared-memory
// data path (128 B a clock per SM) is not taken by the two permutations and by moving the
// vector between the butterfly levels.  Hence:
//  * Each thread keeps E = 2^LE entries in registers (E = 64 for r >= 11), so that the r
//    levels take two register passes with one exchange through shared memory between them,
//    and no lane shuffles (one or two levels of them for r = 7, 13, 14).
//  * Both permutations are free of bank conflicts.  Sample n is copied (cp.async) to a slot of
//    the row's buffer that the host has chosen: the 16 slots of line s >> 4 hold the 16
//    entries that a half-warp reads together, in an order such that the 16 consecutive
//    samples that a half-warp writes together also lie in 16 different bank pairs.  Such an
//    order exists for any permutation (the entries are the edges of a 16-regular bipartite
//    multigraph between write groups and read groups, which 16 colours colour properly) and
//    is found by four halvings of the graph.  The same on the way out.  Addressed by s itself,
//    the scatter and the gather each took about 3 wavefronts for every one they need.
//    (With the r <= 8 levels of a pass done by lane shuffles and X addressed by s, 512 frames x
//    128 rows of N = 4095 with 2048 lags took 0.93 ms; without, 0.67 ms.)
//  * A team of G = 2^r / E threads (one warp or less for r <= 11) owns a row; teams only
//    synchronise within themselves, so the rows of an SM sit in different phases and the
//    loads of some overlap the additions of others.  The registers and the buffer of a team
//    hold one row only, so it asks L2 for its next row while it works on this one: its load
//    phase then waits for L2, not for memory.  65536 rows of N = 4095, 2048 lags: 0.68 -> 0.56
//    ms (5.7 TB/s); 131072 rows of N = 1023, 512 lags: 277 -> 248 us (6.5 TB/s, 0.95 of a copy).
// Against the dense sum (pnce_simt.cu): N = 4095, 2048 lags, 65536 rows 34.4 -> 0.56 ms;
// N = 1023, 512 lags, 8192 rows 0.283 -> 0.028 ms; and closer to the 64-bit result (relative
// error 0.7-1.0e-7 where the dense sum has 5e-7-1.1e-6: fewer roundings per output).
#include <stdlib.h>

#include <algorithm>
#include <new>
#include <utility>
#include <vector>

#include "pnce_mst.h"
#include "pnce_quant.h"

namespace {

// Entries per thread for degree r
constexpr int mst_le(int r) {
    return r >= 11 ? 6 : r >= 9 ? 5 : r == 8 ? 4 : 3;
}

template <int R>
struct Mst {
    static constexpr int LE = mst_le(R), E = 1 << LE;
    static constexpr int LG = R - LE, G = 1 << LG;       // threads per row
    static constexpr int L2 = LG < LE ? LG : LE;         // levels of the second register pass
    static constexpr int X = LG > LE ? LG - LE : 0;      // levels by lane shuffles
    static constexpr int S = 1 << R;
    static constexpr int TEAM = G < 32 ? 32 : G;         // threads that synchronise
    static constexpr int RT = TEAM / G;                  // rows per team
    static constexpr int ROW = S + (S >> L2);            // entries of a row's buffer, padded
    // tables in shared memory; for r >= 13 they are read from global memory
    static constexpr bool TAB_SMEM = R <= 12;
    static constexpr int TAB = TAB_SMEM ? (S * 6 + S / 2 + 127) / 128 * 128 : 0;
    static constexpr int TAB_FEW = TAB_SMEM ? (S * 2 + S / 2 + 127) / 128 * 128 : 0;   // of FEW
    // most threads per block and most blocks per SM (registers: 2 E + about 40 each)
    static constexpr int MAXT = R >= 14 ? 256 : R >= 11 ? 384 : R >= 9 ? 640 : 512;
    static constexpr int MINB = R >= 9 ? 1 : 2;
    static_assert(ROW * sizeof(float2) % 128 == 0, "row buffers are 128-byte aligned");
    static constexpr size_t team_bytes() { return (size_t)RT * ROW * sizeof(float2); }
};

// entry of register k of thread t in the second pass
__host__ __device__ constexpr int pass2_entry(int le, int lg, int t, int k) {
    return lg <= le ? ((t + ((k >> lg) << lg)) << lg) | (k & ((1 << lg) - 1))
                    : (t << le) | k;
}

template <int TEAM>
__device__ __forceinline__ void team_sync(int team) {
    if constexpr (TEAM <= 32)
        __syncwarp();
    else
        asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(TEAM) : "memory");
}

__device__ __forceinline__ void cp_async8(unsigned smem, const void* gmem, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem), "l"(gmem),
                 "r"(bytes)
                 : "memory");
}

// asks for the 16-byte units that lie within n samples
__device__ __forceinline__ void prefetch_l2(const float2* row, int n) {
    const uintptr_t a = ((uintptr_t)row + 15) & ~(uintptr_t)15;
    const unsigned bytes = (unsigned)((uintptr_t)(row + n) - a) & ~15u;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(bytes) : "memory");
}

// the largest magnitude; a NaN is left out
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// butterfly levels on register distances FIRST, 2 FIRST, .. < LAST
template <int E, int FIRST, int LAST>
__device__ __forceinline__ void butterflies(float2 (&v)[E]) {
    const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int d = FIRST; d < LAST; d <<= 1) {
#pragma unroll
        for (int k = 0; k < E; ++k) {
            if (k & d) continue;
            const float2 a = v[k], b = v[k + d];
            v[k] = __fadd2_rn(a, b);
            v[k + d] = __ffma2_rn(b, m1, a);       // a - b, rounded once
        }
    }
}

// v = round(v 2^s) in the format, s from the row's peak
template <int DT, int E>
__device__ __forceinline__ void round_entries(float2 (&v)[E], float sc) {
#pragma unroll
    for (int k = 0; k < E; ++k)
        v[k] = pnce::round_through<DT>(make_float2(v[k].x * sc, v[k].y * sc));
}

// The same for fp16 and e4m3 where no |v 2^s| rounds above the format's largest number, in
// FP32 arithmetic: adding and taking away 1.5 x 2^(e + D), e the exponent of v 2^s but not less
// than the format's smallest, leaves v 2^s rounded to even at the format's last place (a NaN
// stays one).  Conversions to and from the formats seem to issue at 16 a clock per SM and held
// the kernel up: 65536 rows of N = 4095, 2048 lags, fp16 0.78 -> 0.65 ms; e4m3, 32768 rows, 0.347
// -> 0.337 ms.  (bf16 and tf32 need one and two conversions per sample.)  Adding and clamping
// the exponent in one instruction, the peak by three-way maxima and the colour or-ed into the
// address of the first pass's reads: 0.643 -> 0.615 ms and 0.336 -> 0.323 ms.
template <int DT, int E>
__device__ __forceinline__ void round_small(float2 (&v)[E], float sc, int se) {
    constexpr int D = DT == PNCE_FP16 ? 13 : 20, EMIN = DT == PNCE_FP16 ? -14 : -6;
    const int add = (D + se) * (1 << 23) + 0x400000, least = (127 + EMIN + D) * (1 << 23) + 0x400000;
    const float2 sc2 = make_float2(sc, sc), m1 = make_float2(-1.f, -1.f);
#pragma unroll
    for (int k = 0; k < E; ++k) {
        const float2 big = make_float2(
            __int_as_float(__viaddmax_s32(__float_as_int(v[k].x) & 0x7f800000, add, least)),
            __int_as_float(__viaddmax_s32(__float_as_int(v[k].y) & 0x7f800000, add, least)));
        v[k] = __ffma2_rn(big, m1, __ffma2_rn(v[k], sc2, big));
    }
}

// The reduced formats (fp16, bf16, e4m3, tf32) take the same kernel: ROUND rounds the samples in
// registers to what the quantiser would store (each value is exact in FP32), so the step is
// one pass over Y with no operand in memory, and the sums keep all FP32 bits that the tensor
// cores truncate.  One pass against quantise + tensor-core correlation: 65536 rows of
// N = 4095, 2048 lags, fp16 1.43 -> 0.615 ms, e4m3 (32768 rows) 0.485 -> 0.32 ms; 8192 rows of
// N = 1023, 512 lags, tf32 60 -> 27 us; relative error of the sums at N = 4095, fp16,
// 1.4e-6 -> 1e-7.  CODES reads an operand that the quantiser has stored (traced calls, the
// separate correlation step): the same bits.
//
// What a row is: FP32 samples (PLAIN), FP32 samples to be rounded to a reduced format first
// (ROUND), or codes that the quantiser has stored (CODES).
enum { PLAIN = 0, ROUND = 1, CODES = 2 };

// A row of stored codes into its buffer: the loads of up to 32 samples first (the registers are
// free at this point), then their conversions; the team's next row is asked of L2.  With the
// format looked up per sample, and so one sample's loads at a time, 65536 rows of N = 4095 with
// 2048 lags took 4.9 ms in fp16; now 0.55
// (e4m3 0.54, bf16 0.55, tf32 0.68).
template <int R, int DT>
__device__ __forceinline__ void load_codes(const pnce::MstLaunch& p, long long row,
                                           long long stride, const uint4* in_slot, float2* buf,
                                           int t) {
    using M = Mst<R>;
    using T = typename pnce::Fmt<DT>::T;
    constexpr int E = M::E, G = M::G, B = E < 32 ? E : 32;
    const char* op = static_cast<const char*>(p.operand);
    const T* re = reinterpret_cast<const T*>(op + pnce::operand_row(row, 0) * p.op_pitch);
    const T* im = reinterpret_cast<const T*>(op + pnce::operand_row(row, 1) * p.op_pitch);
    if (t < 2 && row + stride < p.A) {
        const void* next = op + pnce::operand_row(row + stride, t) * p.op_pitch;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(next),
                     "r"((unsigned)p.op_pitch) : "memory");
    }
#pragma unroll
    for (int b = 0; b < E; b += B) {
        T cr[B], ci[B];
#pragma unroll
        for (int e = 0; e < B; ++e) {              // (rows are padded: sample N can be read)
            cr[e] = __ldg(re + t + G * (b + e));
            ci[e] = __ldg(im + t + G * (b + e));
        }
#pragma unroll
        for (int e8 = 0; e8 < B; e8 += 8) {
            const uint4 q = in_slot[(b + e8) / 8 * G + t];
            const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                float2 x = pnce::decode<DT>(cr[e8 + e], ci[e8 + e]);
                if (b + e8 + e == E - 1 && t + G * (E - 1) >= p.N)
                    x = make_float2(0.f, 0.f);     // entry 0 of X is zero
                buf[(e & 1) ? w[e / 2] >> 16 : w[e / 2] & 0xffffu] = x;
            }
        }
    }
}

// Few lags (FEW): the second pass and the exchange before it would form all 2^r sums for a
// handful.  Instead the registers' sums V_t[k] of the wanted rows k (the upper bits of the
// columns' vectors u_j: at most one row per column) are left in the buffer, and P threads per
// column add its G = 2^r / E values with their signs.  Taken for up to few_cols columns, where it
// is the faster one, in us, with / without (1.07 GB of samples each, whatever r):
//   r    12: 16 columns 181 / 231, 32 211 / 231, 48 268 / 231
//        11: 16 173 / 208, 32 201 / 208, 48 223 / 208     10: 16 178 / 189, 32 258 / 191
//         9: 8 169 / 188, 16 204 / 198     8: 8 173 / 191, 16 235 / 200     7: 8 218 / 249
// Against one bit test and one addition per sample and lag (pnce_simt.cu), same sizes: r = 12,
// 16 lags 253 -> 181, 8 lags 182 -> 174; r = 10, 16 lags 298 -> 178; r = 7, 8 lags 546 -> 218;
// relative error 5.8-8.9e-8 -> 4.6-7.9e-8.
// A batch's rows of as few lags take the same form, so that a request has the bits of an estimate
// of its own in any mix; the other rows of the batch take the second pass.
constexpr int few_cols(int r) { return r >= 11 ? 32 : r == 10 ? 16 : 8; }

// P = 2^lg_parts: as many threads per column as a row's G allow, 32 at most
__host__ __device__ constexpr int lg_parts_of(int cols, int G) {
    int lg = 0;
    while (lg < 5 && (cols << (lg + 1)) <= G) ++lg;
    return lg;
}

// G (a power of two) values of one column: sum over t of (-1)^<ul, t> V_t, the P = 2^lgP
// threads of the column taking every P-th each; the same on all P lanes.  row: V_t at
// (t + rot) mod G.  lanes: those of the warp that are here.
template <int G>
__device__ __forceinline__ float2 column_sum(const float2* row, int rot, unsigned ul, int part,
                                             int lgP, unsigned lanes) {
    const int n = G >> lgP;
    float2 acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = make_float2(0.f, 0.f);
    for (int i0 = 0; i0 < n; i0 += 32) {
        // bit i: the sign of value part + P (i0 + i)
        const unsigned x = ul >> lgP;
        unsigned w = (__popc(ul & (unsigned)(part + (i0 << lgP))) & 1) ? 0xffffffffu : 0u;
        w ^= (x & 1u ? 0xaaaaaaaau : 0u) ^ (x & 2u ? 0xccccccccu : 0u) ^ (x & 4u ? 0xf0f0f0f0u : 0u) ^
             (x & 8u ? 0xff00ff00u : 0u) ^ (x & 16u ? 0xffff0000u : 0u);
        const int m = n < 32 ? n : 32;
        for (int i = 0; i < m; i += 8) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (e < m) {
                    const float2 v = row[(part + ((i0 + i + e) << lgP) + rot) & (G - 1)];
                    const float sg = __uint_as_float((w << (31 - e) & 0x80000000u) | 0x3f800000u);
                    acc[e] = __ffma2_rn(v, make_float2(sg, sg), acc[e]);
                }
            }
            w >>= 8;
        }
    }
#pragma unroll
    for (int d = 4; d; d >>= 1)
#pragma unroll
        for (int e = 0; e < d; ++e) acc[e] = __fadd2_rn(acc[e], acc[e + d]);
    float2 s = acc[0];
    for (int o = 1; o < (1 << lgP); o <<= 1)
        s = __fadd2_rn(s, make_float2(__shfl_xor_sync(lanes, s.x, o),
                                      __shfl_xor_sync(lanes, s.y, o)));
    return s;
}

// The columns of a row whose V_t[k] lie in the buffer, [k][(t + 4 k) mod G] (lanes of different
// columns, 4 or more neighbours of each, mostly meet different bank pairs)
template <int G, int LG>
__device__ __forceinline__ void few_columns(const float2* buf, const uint16_t* u_of, int cols,
                                            int lgP, int t, float scale, float2* h,
                                            unsigned lanes) {
    for (int c0 = 0; c0 < cols; c0 += G >> lgP) {
        const int part = t & ((1 << lgP) - 1), c = c0 + (t >> lgP);
        const unsigned u = u_of[c < cols ? c : 0], k = u >> LG;
        const float2 w =
            column_sum<G>(buf + k * G, (int)(4 * k), u & (G - 1), part, lgP, lanes);
        if (h && part == 0 && c < cols) h[c] = make_float2(w.x * scale, w.y * scale);
    }
}

// column k L + l holds lag k step + l
__device__ __forceinline__ int lag_of(const pnce::MstLaunch& p, int c) {
    if (p.lags.mode == 0) return c;
    const int k = (int)__umulhi((unsigned)c << 4, p.magic_L);
    return k * p.lags.step + (c - k * p.lags.L);
}

// Where the rows are: one array (ROWS), or a serving batch's requests, described by tables in
// device memory that another kernel has checked (TABLE), or by the launch's parameters (LIST).
enum { ROWS = 0, TABLE = 1, LIST = 2 };

template <int R, int IO, int MODE, bool FEW>
__device__ __forceinline__ void mst_rows(const pnce::MstLaunch& p, const pnce::MstBatch* q) {
    using M = Mst<R>;
    constexpr int E = M::E, G = M::G, LG = M::LG, LE = M::LE, S = M::S;
    extern __shared__ __align__(128) unsigned char mst_smem[];
    const int tid = threadIdx.x;
    uint16_t u_tid = 0;                          // (its load overlaps those of the tables)
    if constexpr (IO != ROWS) {
        if (tid < few_cols(R)) u_tid = __ldg(p.lagvec + tid);      // a block has 32 threads or more
    }
    const uint16_t* tab;
    if constexpr (M::TAB_SMEM) {
        const uint4* src = reinterpret_cast<const uint4*>(p.tab);
        uint4* dst = reinterpret_cast<uint4*>(mst_smem);
        if constexpr (FEW) {
            for (int i = tid; i < (S * 2 + S / 2) / 16; i += blockDim.x)
                dst[i] = __ldg(src + (i < S / 8 ? i : i + S / 4));
        } else {
            for (int i = tid; i < (S * 6 + S / 2) / 16; i += blockDim.x) dst[i] = __ldg(src + i);
        }
        tab = reinterpret_cast<const uint16_t*>(mst_smem);
    } else {
        tab = p.tab;
    }
    __shared__ uint16_t few_u[few_cols(R)];      // u_j of the columns
    __shared__ unsigned few_rows[2];               // rows k that they need
    if constexpr (FEW) {
        if (tid < 2) few_rows[tid] = 0;
        __syncthreads();
        for (int c = tid; c < p.lags.ldH; c += blockDim.x) {
            const unsigned u = __ldg(p.lagvec + lag_of(p, c));
            few_u[c] = (uint16_t)u;
            atomicOr(&few_rows[u >> LG >> 5], 1u << (u >> LG & 31));
        }
    } else if constexpr (IO != ROWS) {
        if (tid < few_cols(R)) few_u[tid] = u_tid;
    }
    if constexpr (M::TAB_SMEM || FEW || IO != ROWS) __syncthreads();
    const uint4* in_slot = reinterpret_cast<const uint4*>(tab);            // [E/8][G] x 8
    const uint4* out_slot = reinterpret_cast<const uint4*>(tab + S);       // [E/8][G] x 8
    const uint16_t* lag_slot = tab + 2 * S;                                // [N]
    const uint32_t* in_col = reinterpret_cast<const uint32_t*>(
        tab + (FEW && M::TAB_SMEM ? 1 : 3) * S);                               // [E/8][G]

    // as a programmatic dependent the tables came in beside the kernel before; everything else
    // is read and written only after it has finished.  Estimates that follow each other in a
    // stream overlap their launches and their last rows this way: 4736 rows of N = 2047, 512 lags
    // 26.8 -> 25.1 us; 8192 rows of N = 1023 22.5 -> 21.9.  (No block of the next grid can keep
    // one of this grid waiting: the grids are no larger than what is resident.)
    if constexpr (IO == ROWS) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (IO != LIST) asm volatile("griddepcontrol.wait;" ::: "memory");
    __shared__ float s_peak[16][8];                // peaks of a team's warps

    const int team = tid / M::TEAM, t = tid % G, sub = (tid % M::TEAM) / G;
    float2* buf = reinterpret_cast<float2*>(mst_smem + (FEW ? M::TAB_FEW : M::TAB)) +
                  (team * M::RT + sub) * M::ROW;
    const unsigned sbuf = (unsigned)__cvta_generic_to_shared(buf);
    const int teams = blockDim.x / M::TEAM;
    const long long stride = (long long)gridDim.x * teams * M::RT;
    if constexpr (R >= 11 && IO == ROWS && MODE != CODES) {
        if (team >= p.late_from) __nanosleep(2200);
    }

    for (long long row0 = ((long long)blockIdx.x * teams + team) * M::RT; row0 < p.A;
         row0 += stride) {
        const long long row = row0 + sub;
        const float2* y = nullptr;
        float2* h = nullptr;
        int cols = p.lags.ldH;
        if (row < p.A) {
            if constexpr (IO == TABLE) {
                const int b = p.row_req[row];     // a plain load: it stays behind the wait
                if (b >= 0) {
                    const pnce_req_desc& d = p.dd[b];
                    cols = d.K * d.L;
                    y = static_cast<const float2*>(d.Y) + (row - d.row_offset) * p.N;
                    h = static_cast<float2*>(d.H) + (row - d.row_offset) * cols;
                }
            } else if constexpr (IO == LIST) {
                int b = 0;                         // the last request that begins at or before row
#pragma unroll
                for (int d = pnce::kMstBatchMax / 2; d; d >>= 1)
                    if (b + d < q->n && q->row0[b + d] <= row) b += d;
                cols = q->cols[b];
                y = q->Y[b] + (row - q->row0[b]) * p.N;
                h = q->H[b] + (row - q->row0[b]) * cols;
            } else {
                y = p.Y + row * p.y_stride;
                h = p.H + row * p.lags.ldH;
            }
        }
        if constexpr (IO == TABLE) {               // a team without a row has nothing to do
            if (M::RT == 1 ? y == nullptr : __all_sync(0xffffffffu, y == nullptr)) continue;
        }
        if constexpr (MODE == CODES) {
            if (row < p.A) {
                switch (p.dtype) {
                    case PNCE_FP16: load_codes<R, PNCE_FP16>(p, row, stride, in_slot, buf, t); break;
                    case PNCE_BF16: load_codes<R, PNCE_BF16>(p, row, stride, in_slot, buf, t); break;
                    case PNCE_TF32: load_codes<R, PNCE_TF32>(p, row, stride, in_slot, buf, t); break;
                    default: load_codes<R, PNCE_FP8E4M3>(p, row, stride, in_slot, buf, t); break;
                }
            }
        } else if (y) {
#pragma unroll
            for (int i8 = 0; i8 < E / 8; ++i8) {
                const uint4 q = in_slot[i8 * G + t];
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int n = t + G * (8 * i8 + e);
                    const unsigned slot = (e & 1) ? w[e / 2] >> 16 : w[e / 2] & 0xffffu;
                    const bool ok = 8 * i8 + e < E - 1 || n < p.N;     // entry 0 of X is zero
                    cp_async8(sbuf + 8 * slot, ok ? y + n : y, ok ? 8 : 0);
                }
            }
        }
        if constexpr (MODE != CODES) asm volatile("cp.async.wait_all;\n" ::: "memory");
        if constexpr (IO == ROWS && MODE != CODES) {
            if (t == 0 && row + stride < p.A) prefetch_l2(y + stride * p.y_stride, p.N);
        }
        team_sync<M::TEAM>(team);

        float2 v[E];
        // first pass: register k holds entry k G + t, levels G .. S/2
#pragma unroll
        for (int k8 = 0; k8 < E / 8; ++k8) {
            const uint32_t c = in_col[k8 * G + t];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int k = 8 * k8 + e;
                // 8 x the colour, or-ed into the address of the line: rows are 128-byte aligned
                const uint32_t off = (e == 0 ? c << 3 : c >> (4 * e - 3)) & 0x78u;
                asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];"
                             : "=f"(v[k].x), "=f"(v[k].y)
                             : "r"(((sbuf + 8 * (t & ~15)) | off) + 8 * G * k)
                             : "memory");
            }
        }
        float scale = p.invN;
        if constexpr (MODE == CODES) {
            if (row < p.A) scale = p.factors[row];
        }
        if constexpr (MODE == ROUND) {
            int se = 0;
            float m = 0.f;
            if (p.target != 0) {                   // NaN parts are left out, as fmaxf does
#pragma unroll
                for (int k = 0; k < E; ++k) m = max3_abs(m, v[k].x, v[k].y);
#pragma unroll
                for (int o = (G < 32 ? G : 32) / 2; o; o >>= 1)
                    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if constexpr (G > 32) {
                    if ((t & 31) == 0) s_peak[team][t >> 5] = m;
                    team_sync<M::TEAM>(team);
#pragma unroll
                    for (int w = 0; w < G / 32; ++w) m = fmaxf(m, s_peak[team][w]);
                }
                se = pnce::scale_exponent(p.target, m);
                scale = ldexpf(p.invN, -se);
            }
            const float sc = ldexpf(1.0f, se);
            const bool small = m * sc < ldexpf(1.0f, p.target);   // no code overflows
            if (p.dtype == PNCE_FP16 && small) {
                round_small<PNCE_FP16>(v, sc, se);
            } else if (p.dtype == PNCE_FP8E4M3 && small) {
                round_small<PNCE_FP8E4M3>(v, sc, se);
            } else {
                switch (p.dtype) {
                    case PNCE_FP16: round_entries<PNCE_FP16>(v, sc); break;
                    case PNCE_BF16: round_entries<PNCE_BF16>(v, sc); break;
                    case PNCE_TF32: round_entries<PNCE_TF32>(v, sc); break;
                    default: round_entries<PNCE_FP8E4M3>(v, sc); break;
                }
            }
        }
        butterflies<E, 1, E>(v);
        team_sync<M::TEAM>(team);                  // the buffer is read: reuse it
        bool few = FEW, second = !FEW;             // forms of this row, and of its team's rows
        if constexpr (FEW) {
            const unsigned rows0 = few_rows[0], rows1 = few_rows[1];
#pragma unroll
            for (int k = 0; k < E; ++k)
                if ((k < 32 ? rows0 : rows1) >> (k & 31) & 1)
                    buf[k * G + ((t + 4 * k) & (G - 1))] = v[k];
            team_sync<M::TEAM>(team);
            few_columns<G, LG>(buf, few_u, cols, p.lg_parts, t, scale, h, 0xffffffffu);
        } else if constexpr (IO != ROWS) {
            few = cols <= few_cols(R);
            if (M::RT == 1 ? few : __any_sync(0xffffffffu, few)) {
                second = M::RT != 1 && __any_sync(0xffffffffu, !few);
#pragma unroll
                for (int k = 0; k < E; ++k) buf[k * G + ((t + 4 * k) & (G - 1))] = v[k];
                team_sync<M::TEAM>(team);
                // the rows of a warp may differ in their columns: each with its own lanes
                const unsigned lanes =
                    G < 32 ? ((1u << (G & 31)) - 1u) << ((tid & 31) & ~(G - 1)) : 0xffffffffu;
                if (few)
                    few_columns<G, LG>(buf, few_u, cols, lg_parts_of(cols, G), t, scale, h, lanes);
                if (second) {                     // (read again: kept, they would not fit)
#pragma unroll
                    for (int k = 0; k < E; ++k) v[k] = buf[k * G + ((t + 4 * k) & (G - 1))];
                    team_sync<M::TEAM>(team);
                }
            }
        }
        if (second) {
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const int s = k * G + t;
                buf[s + (s >> M::L2)] = v[k];
            }
            team_sync<M::TEAM>(team);
            // second pass: the low L2 levels in registers, the X above them by lane shuffles
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const int s = pass2_entry(LE, LG, t, k);
                v[k] = buf[s + (s >> M::L2)];
            }
            butterflies<E, 1, (1 << M::L2)>(v);
            if constexpr (M::X > 0) {
#pragma unroll
                for (int d = 1; d < (1 << M::X); d <<= 1) {
                    const float sg = (t & d) ? -1.f : 1.f;
#pragma unroll
                    for (int k = 0; k < E; ++k) {
                        const float px = __shfl_xor_sync(0xffffffffu, v[k].x, d);
                        const float py = __shfl_xor_sync(0xffffffffu, v[k].y, d);
                        v[k] = make_float2(fmaf(sg, v[k].x, px), fmaf(sg, v[k].y, py));
                    }
                }
            }
            team_sync<M::TEAM>(team);
            // out: only the lines of lags that are wanted (contiguous lags), all of them otherwise
            const unsigned lim = p.lags.mode == 0 ? (unsigned)((cols + 15) & ~15) : (unsigned)S;
#pragma unroll
            for (int k8 = 0; k8 < E / 8; ++k8) {
                const uint4 q = out_slot[k8 * G + t];
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const unsigned slot = (e & 1) ? w[e / 2] >> 16 : w[e / 2] & 0xffffu;
                    if (slot < lim) buf[slot] = v[8 * k8 + e];
                }
            }
            team_sync<M::TEAM>(team);
            if (h && !few) {
                for (int c = t; c < cols; c += G) {
                    const int lag = IO != ROWS ? c : lag_of(p, c);
                    const float2 w = buf[lag_slot[lag]];
                    h[c] = make_float2(w.x * scale, w.y * scale);
                }
            }
        }
        team_sync<M::TEAM>(team);                  // the buffer takes the next row
    }
}

template <int R, int IO, int MODE, bool FEW>
__global__ void __launch_bounds__(Mst<R>::MAXT, Mst<R>::MINB)
mst_kernel(const __grid_constant__ pnce::MstLaunch p) {
    mst_rows<R, IO, MODE, FEW>(p, nullptr);
}

template <int R, int MODE>
__global__ void __launch_bounds__(Mst<R>::MAXT, Mst<R>::MINB)
mst_batch_kernel(const __grid_constant__ pnce::MstLaunch p,
                 const __grid_constant__ pnce::MstBatch q) {
    mst_rows<R, LIST, MODE, false>(p, &q);
}

using MstKernel = void (*)(const pnce::MstLaunch);
using MstBatchKernel = void (*)(const pnce::MstLaunch, const pnce::MstBatch);

template <int R, bool FEW>
MstKernel estimate_kernel(int mode) {
    return mode == PLAIN   ? mst_kernel<R, ROWS, PLAIN, FEW>
           : mode == ROUND ? mst_kernel<R, ROWS, ROUND, FEW>
                           : mst_kernel<R, ROWS, CODES, FEW>;
}

template <int R>
MstKernel kernel_of(bool table, int mode, bool few) {
    if (table)
        return mode == ROUND ? mst_kernel<R, TABLE, ROUND, false>
                             : mst_kernel<R, TABLE, PLAIN, false>;
    return few ? estimate_kernel<R, true>(mode) : estimate_kernel<R, false>(mode);
}

template <int R>
MstBatchKernel batch_kernel_of(int mode) {
    return mode == ROUND ? mst_batch_kernel<R, ROUND> : mst_batch_kernel<R, PLAIN>;
}

}  // namespace

namespace pnce {

// Teams that start together load together and then add together.  Where a row is several
// microseconds of work (r >= 11), each team has two or more and a block has several, half of a
// block's teams (r = 13: two of three) start 2 us later: the other half's first rows still keep the
// memory busy, and from then on one half loads while the other adds.  us without / with: N = 2047,
// 4736 rows of 4 x 128 spread lags 31.7 / 29.8, 5473 rows of 1024 lags 32.0 / 29.6; N = 4095, 65536
// rows of 2048 lags 552 / 545, fp16 615 / 606, 2737 rows 34.8 / 32.1, 32768 rows of 16 lags 177.5 /
// 174.2 (1.5 to 5 us are alike); N = 8191, 913 rows 43.9 / 41.8, 4000 rows 121.1 / 116.0 (one late
// team of three: 43.2, 118.7).  Shorter rows lose: N = 1023 fp16 1 %, N = 127 with 5 lags 5-13 %.  A
// block of one team (r = 14) has no other half, N = 16383, 304 rows 20.4 / 20.8, fp16, 608 rows 43.8 /
// 45.2, nor do launches from host memory that keep one team per SM in flight (256 rows of N = 4095
// 67.5 / 69.7).
int mst_late_from(int r, int teams, bool two_rounds) {
    return r >= 11 && teams > 1 && two_rounds ? teams / 2 : teams;
}

}  // namespace pnce

namespace {

template <int R>
cudaError_t launch_r(const pnce::MstTables& m, pnce::MstLaunch& p, cudaStream_t s) {
    using M = Mst<R>;
    const bool few = p.lagvec && !p.dd && !p.batch && p.lags.ldH <= few_cols(R);
    p.lg_parts = lg_parts_of(p.lags.ldH, M::G);
    // rows spread over the SMs first, then over the teams of a block
    const long long teams = (p.A + M::RT - 1) / M::RT;
    const long long sms = m.num_sms;
    long long most = teams;                      // teams that work at once
    if (p.in_flight) {
        const long long bytes = (long long)M::RT * p.N * 8;
        most = (p.in_flight + bytes - 1) / bytes;
        if (most < sms) most = sms;
        if (most > teams) most = teams;
    }
    long long per = (most + sms - 1) / sms;
    if (per > m.block_teams) per = m.block_teams;
    long long grid = (teams + per - 1) / per;
    const long long resident = sms * (per == m.block_teams ? m.blocks_per_sm : 1);
    if (grid > resident) grid = resident;
    if (p.in_flight && grid > (most + per - 1) / per) grid = (most + per - 1) / per;
    p.late_from = pnce::mst_late_from(R, (int)per, 2 * grid * per * M::RT <= p.A);
    const int mode = p.operand ? CODES : p.dtype != PNCE_FP32_SIMT ? ROUND : PLAIN;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3((unsigned)(per * M::TEAM), 1, 1);
    cfg.dynamicSmemBytes = (few ? M::TAB_FEW : M::TAB) + (size_t)per * M::team_bytes();
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = p.pdl || !(p.dd || p.batch) ? 1 : 0;
    if (p.batch) return cudaLaunchKernelEx(&cfg, batch_kernel_of<R>(mode), p, *p.batch);
    return cudaLaunchKernelEx(&cfg, kernel_of<R>(p.dd != nullptr, mode, few), p);
}

// Shared-memory limits of the kernels, and how many teams fit an SM.
template <int R>
cudaError_t setup_r(pnce::MstTables& m, int max_smem_optin) {
    using M = Mst<R>;
    int teams = M::MAXT / M::TEAM;
    const int fit = (int)((max_smem_optin - M::TAB) / M::team_bytes());
    if (fit < 1) return cudaErrorNotSupported;
    if (teams > fit) teams = fit;
    const int smem = M::TAB + teams * (int)M::team_bytes();
    cudaError_t e;
    for (int i = 0; i < 8; ++i) {                // plain, rounding, codes, (serving: two); few
        const int mode = i % 4 == 3 ? (i == 3 ? (int)PLAIN : (int)ROUND) : i % 4;
        if ((e = cudaFuncSetAttribute(kernel_of<R>(i % 4 == 3, mode, i >= 4),
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) !=
            cudaSuccess)
            return e;
    }
    for (int mode : {(int)PLAIN, (int)ROUND})
        if ((e = cudaFuncSetAttribute(batch_kernel_of<R>(mode),
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) !=
            cudaSuccess)
            return e;
    m.block_teams = teams;
    int per = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel_of<R>(false, PLAIN, false),
                                                           teams * M::TEAM, smem)) != cudaSuccess)
        return e;
    m.blocks_per_sm = per < 1 ? 1 : per;
    return cudaSuccess;
}

// Proper 16-colouring of a 16-regular bipartite multigraph given as edges (l[e], r[e]),
// e < S, both sides of S / 16 vertices: four times, the edges of a class are split into two
// classes of half the degree by pairing them up at every vertex and colouring the cycles that
// the pairs form alternately.
void colour16(const std::vector<int>& l, const std::vector<int>& r, std::vector<uint8_t>& col) {
    const int S = (int)l.size(), V = S / 16;
    col.assign((size_t)S, 0);
    std::vector<int> pl((size_t)S + 1), pr((size_t)S + 1), open((size_t)V * 16);
    std::vector<int8_t> half((size_t)S);
    for (int level = 0; level < 4; ++level) {
        for (int side = 0; side < 2; ++side) {
            const std::vector<int>& v = side ? r : l;
            std::vector<int>& p = side ? pr : pl;
            std::fill(open.begin(), open.end(), -1);
            for (int e = 0; e < S; ++e) {          // (no branch: it would be a coin toss)
                int& o = open[(size_t)v[(size_t)e] * 16 + col[(size_t)e]];
                const int first = o;
                p[(size_t)e] = first;              // the first of a pair: set by the second
                p[(size_t)(first < 0 ? S : first)] = e;
                o = first < 0 ? e : -1;
            }
        }
        std::fill(half.begin(), half.end(), (int8_t)-1);
        for (int e0 = 0; e0 < S; ++e0)
            for (int e = e0; half[(size_t)e] < 0; e = pr[(size_t)pl[(size_t)e]]) {
                half[(size_t)e] = 0;
                half[(size_t)pl[(size_t)e]] = 1;
            }
        for (int e = 0; e < S; ++e)
            col[(size_t)e] = (uint8_t)(2 * col[(size_t)e] + half[(size_t)e]);
    }
}

}  // namespace

namespace pnce {

size_t mst_table_bytes(int N) {
    int r = 0;
    while ((1LL << r) < (long long)N + 1) ++r;
    if ((1LL << r) != (long long)N + 1 || r < kMstMinR || r > kMstMaxR) return 0;
    return (size_t)(N + 1) * 13 / 2;
}

bool mst_build_tables(const uint32_t* bits_host, int N, uint16_t* out) {
    return mst_build_tables(bits_host, N, out, nullptr);
}

bool mst_build_tables(const uint32_t* bits_host, int N, uint16_t* out, uint16_t* lagvec) {
    if (mst_table_bytes(N) == 0) return false;
    int r = 0;
    while ((1 << r) < N + 1) ++r;
    const int S = 1 << r, le = mst_le(r), lg = r - le, E = 1 << le, G = 1 << lg;
    std::vector<uint16_t> pos((size_t)N), lag((size_t)N);
    if (pnce_fmt_tables(bits_host, N, pos.data(), lag.data()) != PNCE_OK) return false;
    if (lagvec) std::copy(lag.begin(), lag.end(), lagvec);
    std::vector<int> l((size_t)S), rr((size_t)S), of((size_t)S);
    std::vector<uint8_t> col;
    uint16_t* in_slot = out;
    uint16_t* out_slot = out + S;
    uint16_t* lag_slot = out + 2 * S;
    uint8_t* in_col = reinterpret_cast<uint8_t*>(out + 3 * S);
    // in: edge n joins write group n >> 4 to read group s_n >> 4 (n = N: entry 0)
    for (int n = 0; n < S; ++n) {
        const int s = n < N ? pos[(size_t)n] : 0;
        l[(size_t)n] = n >> 4;
        rr[(size_t)n] = s >> 4;
    }
    colour16(l, rr, col);
    for (int n = 0; n < S; ++n) {
        const int s = n < N ? pos[(size_t)n] : 0;
        const int i = n >> lg, t = n & (G - 1);
        in_slot[((i / 8) * G + t) * 8 + i % 8] = (uint16_t)((s & ~15) | col[(size_t)n]);
        of[(size_t)s] = col[(size_t)n];
    }
    for (int t = 0; t < G; ++t)
        for (int k = 0; k < E; k += 2)
            in_col[4 * ((k / 8) * G + t) + (k % 8) / 2] =
                (uint8_t)(of[(size_t)(k * G + t)] | (of[(size_t)((k + 1) * G + t)] << 4));
    // out: edge j joins the half-warp that holds entry u_j to read group j >> 4
    std::vector<int> half_of((size_t)S);
    for (int t = 0; t < G; ++t)
        for (int k = 0; k < E; ++k)
            half_of[(size_t)pass2_entry(le, lg, t, k)] = k * (G / 16) + (t >> 4);
    std::fill(of.begin(), of.end(), N);                       // lag of an entry (0: none)
    for (int j = 0; j < N; ++j) of[lag[(size_t)j]] = j;
    for (int j = 0; j < S; ++j) {
        l[(size_t)j] = half_of[j < N ? lag[(size_t)j] : 0];
        rr[(size_t)j] = j >> 4;
    }
    colour16(l, rr, col);
    for (int j = 0; j < S; ++j) lag_slot[j] = (uint16_t)((j & ~15) | col[(size_t)j]);
    for (int t = 0; t < G; ++t)
        for (int k = 0; k < E; ++k)
            out_slot[((k / 8) * G + t) * 8 + k % 8] =
                lag_slot[of[(size_t)pass2_entry(le, lg, t, k)]];
    return true;
}

cudaError_t mst_setup(MstTables& m, const uint16_t* tab_dev, int N, int num_sms,
                      int max_smem_optin) {
    m.tab = nullptr;
    m.lagvec = nullptr;
    m.N = N;
    m.num_sms = num_sms;
    m.r = 0;
    while ((1 << m.r) < N + 1) ++m.r;
    cudaError_t e = cudaErrorInvalidValue;
    switch (m.r) {
        case 7: e = setup_r<7>(m, max_smem_optin); break;
        case 8: e = setup_r<8>(m, max_smem_optin); break;
        case 9: e = setup_r<9>(m, max_smem_optin); break;
        case 10: e = setup_r<10>(m, max_smem_optin); break;
        case 11: e = setup_r<11>(m, max_smem_optin); break;
        case 12: e = setup_r<12>(m, max_smem_optin); break;
        case 13: e = setup_r<13>(m, max_smem_optin); break;
        case 14: e = setup_r<14>(m, max_smem_optin); break;
        default: break;
    }
    if (e == cudaSuccess) m.tab = tab_dev;
    return e;
}

bool mst_replaces_tc(const pnce_pilot* pilot) {
    if (!pilot->mst.tab) return false;
    for (const char* name : {"PNCE_TC_PAIRS", "PNCE_TC_STAGED_PILOT", "PNCE_TC_LAGMAJOR",
                             "PNCE_TC_LAGMAJOR_CL", "PNCE_TC_SMALL_GRID_BN",
                             "PNCE_TC_TEST_DROP_ARRIVE", "PNCE_TC_FORCE"})
        if (getenv(name)) return false;
    return true;
}

cudaError_t launch_mst(const MstTables& m, MstLaunch p, cudaStream_t s) {
    if (p.A <= 0) return cudaSuccess;
    p.target = p.dtype == PNCE_FP16      ? Fmt<PNCE_FP16>::target
               : p.dtype == PNCE_FP8E4M3 ? Fmt<PNCE_FP8E4M3>::target
                                         : 0;
    p.op_pitch = (long long)row_pitch(m.N) * elem_bytes(p.dtype);
    p.tab = m.tab;
    p.lagvec = m.lagvec;
    p.N = m.N;
    p.invN = (float)(1.0 / (double)m.N);
    // c / L for c < 2^14 and L < 2^14 as the high word of 16 c * magic_L
    p.magic_L = p.lags.mode ? (unsigned)(((1u << 28) + (unsigned)p.lags.L - 1) / (unsigned)p.lags.L)
                            : 0u;
    switch (m.r) {
        case 7: return launch_r<7>(m, p, s);
        case 8: return launch_r<8>(m, p, s);
        case 9: return launch_r<9>(m, p, s);
        case 10: return launch_r<10>(m, p, s);
        case 11: return launch_r<11>(m, p, s);
        case 12: return launch_r<12>(m, p, s);
        case 13: return launch_r<13>(m, p, s);
        case 14: return launch_r<14>(m, p, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pnce
