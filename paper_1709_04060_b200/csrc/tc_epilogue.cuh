// Epilogue shared by the tcgen05 kernels: accumulators out of tensor memory, the threshold count
// T(x, t) of Section 2.1.1, codes packed and stored.
#pragma once

#include "common.cuh"

namespace qnn {

enum { OUT_RAW = 0, OUT_U8 = 1, OUT_PLANES = 2 };

// ------------------------------------------------------------------- epilogue
// T(x, t) = #{q : t_q <= x}.  When every |acc| is below 2^22 the count runs on the
// FP32 pipe (twice the int32 rate, no conversions): the int32 accumulator x is
// turned into the float 1.5*2^23 + x by one integer add on its bit pattern, each
// threshold is held as the float 1.5*2^23 + (t - 1), and for integers
// saturate((1.5*2^23 + x) - (1.5*2^23 + t - 1)) is exactly 1 if x >= t, else 0.
// Thresholds are clamped to [-2^22 + 1, 2^22] first, which cannot change a
// comparison with such an accumulator.  Counts of two neighbouring channels are
// accumulated in one float on top of 1.5*2^23 (the second scaled by 256), so the
// two codes are the low two bytes of the sum's bit pattern.
// Below 2^24 (8-bit first layers: 363 x 128 x 255) the accumulator is converted instead (exact) and
// compared with the float t - 1: their difference is exact where it is small, and where it is rounded
// it is far outside [0, 1], so the saturated value is the same 0 or 1.
enum { COUNT_INT = 0, COUNT_MAGIC = 1, COUNT_FLOAT = 2 };
constexpr float FP_MAGIC = 12582912.0f;        // 1.5 * 2^23, bit pattern 0x4B400000
constexpr int FP_MAGIC_BITS = 0x4B400000;
constexpr int FP_LIMIT = 1 << 22, FP_LIMIT_FLOAT = 1 << 24;

// How accumulators of magnitude up to K * wmax * amax are counted (wide: by a kernel that has COUNT_FLOAT).
inline int count_mode(double most, bool wide) { return most < double(FP_LIMIT) ? COUNT_MAGIC : (wide && most < double(FP_LIMIT_FLOAT) ? COUNT_FLOAT : COUNT_INT); }

// thresholds per channel in shared memory, padded to a multiple of four
__host__ __device__ constexpr int thr_slots(int out_bits) {
    return out_bits <= 0 ? 4 : (((1 << out_bits) - 1 + 3) / 4 * 4);
}

__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, int (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr) : "memory");
}
// Completes every tcgen05.ld issued so far; the registers pass through the statement so
// that no use of them can be scheduled ahead of it.
__device__ __forceinline__ void tmem_ld_wait(int (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
          "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
          "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
          "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
        :: "memory");
}

// Bits b, 8+b, 16+b, 24+b of x gathered into the low nibble.
__device__ __forceinline__ uint32_t nibble_of_plane(uint32_t x, int b) {
    return (((x >> b) & 0x01010101u) * 0x01020408u) >> 24;
}

// Stage the thresholds of channels [c0, c0 + bn) in shared memory (one warp, a lane per
// channel).  Slots past the row's thresholds and channels past M hold a value no
// accumulator reaches.  Sets of 7 or 15 thresholds are sorted so that the epilogue can
// count by bisection (raw int32); sets of 1 or 3 are counted linearly, in float form
// when the FP count applies.
template <int OUT_BITS, bool SORT = (OUT_BITS >= 3), bool WIDE = false, typename Params>
__device__ __forceinline__ void stage_thresholds(const Params &p, int *thr_s, int c0, int bn, int lane) {
    constexpr int N_THR = (1 << OUT_BITS) - 1, NT = thr_slots(OUT_BITS);
    for (int c = lane; c < bn; c += 32) {
        const int m = c0 + c;
        int t[NT];
#pragma unroll
        for (int q = 0; q < NT; ++q) t[q] = 0x7fffffff;
        if (m < p.M) {
#pragma unroll
            for (int q = 0; q < N_THR; ++q) t[q] = ld_global(p.thr + (size_t)m * N_THR + q);
        }
        if (SORT) {
            // odd-even transposition sort; the pads are the largest value and stay last
#pragma unroll
            for (int r = 0; r < NT; ++r)
#pragma unroll
                for (int i = r & 1; i + 1 < NT; i += 2) {
                    const int lo = min(t[i], t[i + 1]), hi = max(t[i], t[i + 1]);
                    t[i] = lo; t[i + 1] = hi;
                }
        }
        if (OUT_BITS <= 2 && p.count != COUNT_INT) {
            const int limit = !WIDE || p.count == COUNT_MAGIC ? FP_LIMIT : FP_LIMIT_FLOAT;
#pragma unroll
            for (int q = 0; q < NT; ++q) {
                const int tc = t[q] <= -limit ? -limit + 1 : (t[q] > limit ? limit : t[q]);
                t[q] = !WIDE || p.count == COUNT_MAGIC ? FP_MAGIC_BITS + (tc - 1) : __float_as_int((float)(tc - 1));
            }
        }
#pragma unroll
        for (int v = 0; v < NT / 4; ++v)
            reinterpret_cast<int4 *>(thr_s + c * NT)[v] = make_int4(t[4 * v], t[4 * v + 1], t[4 * v + 2], t[4 * v + 3]);
    }
}

// Codes of 32 channels with 1 or 3 thresholds, counted on the FP32 pipe: one float4 of thresholds per
// channel (MAGIC: COUNT_MAGIC, else COUNT_FLOAT).  UNARY: not the count but a bit per threshold.
template <int N_THR, bool MAGIC, bool UNARY>
__device__ __forceinline__ void count_chunk_float(const int *thr_c, const int (&acc)[32], uint32_t (&packed)[8]) {
    auto to_float = [](int x) { return MAGIC ? __int_as_float(x + FP_MAGIC_BITS) : (float)x; };
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        float4 t[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = *reinterpret_cast<const float4 *>(thr_c + (8 * g + e) * 4);
        uint32_t pr[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float x0 = to_float(acc[8 * g + 2 * h]), x1 = to_float(acc[8 * g + 2 * h + 1]);
            const float4 t0 = t[2 * h], t1 = t[2 * h + 1];
            float s0 = __saturatef(x0 - t0.x), s1 = __saturatef(x1 - t1.x);
            if (N_THR > 1) {
                s0 = fmaf(__saturatef(x0 - t0.y), UNARY ? 2.f : 1.f, s0); s1 = fmaf(__saturatef(x1 - t1.y), UNARY ? 2.f : 1.f, s1);
                s0 = fmaf(__saturatef(x0 - t0.z), UNARY ? 4.f : 1.f, s0); s1 = fmaf(__saturatef(x1 - t1.z), UNARY ? 4.f : 1.f, s1);
            }
            pr[h] = (uint32_t)__float_as_int(fmaf(s1, 256.f, s0 + FP_MAGIC));
        }
        packed[2 * g] = __byte_perm(pr[0], pr[1], 0x5410);
        packed[2 * g + 1] = __byte_perm(pr[2], pr[3], 0x5410);
    }
}

// Codes of 32 channels, four to a word.  WIDE: COUNT_FLOAT is among the ways to count.  UNARY (1 or 3 thresholds): a bit per threshold instead, which for
// sorted thresholds is the code in unary: the maximum of such codes is their OR.
template <int OUT_BITS, bool UNARY = false, bool WIDE = false, typename Params>
__device__ __forceinline__ void count_chunk(const Params &p, const int *thr_c, const int (&acc)[32], uint32_t (&packed)[8]) {
    constexpr int N_THR = (1 << OUT_BITS) - 1, NT = thr_slots(OUT_BITS);
    // Eight channels at a time, written so that the threshold loads of all eight are issued
    // before any of them is used (independent chains interleave instead of running one
    // after the other).
    if (OUT_BITS >= 3) {
        // bisection over the channel's sorted thresholds: the row of NT words sits in NT
        // distinct banks, so lanes that look at different slots do not conflict
        // Sixteen channels' searches advance together: a probe's load takes 100+ cycles while the
        // tensor pipe reads shared memory, and only independent chains hide that.
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            // the search position is carried as a pointer (row + count): every probe is a load at a
            // constant offset from it, and a step is load, compare, conditional add
            const int *pos[16];
            int c[16], t[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) pos[e] = thr_c + (16 * g + e) * NT;
#pragma unroll
            for (int step = NT / 2; step >= 1; step >>= 1) {
#pragma unroll
                for (int e = 0; e < 16; ++e) t[e] = pos[e][step - 1];
#pragma unroll
                for (int e = 0; e < 16; ++e) pos[e] += (acc[16 * g + e] >= t[e]) ? step : 0;
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) c[e] = (int)(pos[e] - (thr_c + (16 * g + e) * NT));
#pragma unroll
            for (int v = 0; v < 4; ++v)
                packed[4 * g + v] = (uint32_t)c[4 * v] | ((uint32_t)c[4 * v + 1] << 8) | ((uint32_t)c[4 * v + 2] << 16) |
                                    ((uint32_t)c[4 * v + 3] << 24);
        }
    } else if (p.count == COUNT_MAGIC) {
        count_chunk_float<N_THR, true, UNARY>(thr_c, acc, packed);
    } else if (WIDE && p.count == COUNT_FLOAT) {
        count_chunk_float<N_THR, false, UNARY>(thr_c, acc, packed);
    } else {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            int4 t[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) t[e] = *reinterpret_cast<const int4 *>(thr_c + (8 * g + e) * NT);
            int c[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int x = acc[8 * g + e];
                c[e] = (x >= t[e].x) ? 1 : 0;
                if (N_THR > 1) c[e] += ((x >= t[e].y) ? (UNARY ? 2 : 1) : 0) + ((x >= t[e].z) ? (UNARY ? 4 : 1) : 0);
            }
            packed[2 * g] = (uint32_t)c[0] | ((uint32_t)c[1] << 8) | ((uint32_t)c[2] << 16) | ((uint32_t)c[3] << 24);
            packed[2 * g + 1] = (uint32_t)c[4] | ((uint32_t)c[5] << 8) | ((uint32_t)c[6] << 16) | ((uint32_t)c[7] << 24);
        }
    }
}

// One chunk: this thread's pixel n, channels mc .. mc+31 (accumulators acc[0..31]).
template <int OUT_MODE, int OUT_BITS, bool WIDE = false, typename Params>
__device__ __forceinline__ void epilogue_chunk(const Params &p, const int *thr_c, const int (&acc)[32],
                                               int n, bool n_ok, int mc) {
    if (OUT_MODE == OUT_RAW) {
        if (!n_ok) return;
        int32_t *o = reinterpret_cast<int32_t *>(p.out) + (size_t)n * p.M + mc;
        if ((p.M & 3) == 0 && mc + 32 <= p.M) {
#pragma unroll
            for (int v = 0; v < 8; ++v)
                reinterpret_cast<int4 *>(o)[v] = make_int4(acc[4 * v], acc[4 * v + 1], acc[4 * v + 2], acc[4 * v + 3]);
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (mc + j < p.M) o[j] = acc[j];
        }
        return;
    }
    uint32_t packed[8];                          // four codes per word, one byte each
    count_chunk<OUT_BITS, false, WIDE>(p, thr_c, acc, packed);
    if (!n_ok) return;
    if (OUT_MODE == OUT_U8) {
        uint8_t *o = reinterpret_cast<uint8_t *>(p.out) + (size_t)n * p.ld_out + mc;
        const int valid = p.ld_out - mc;         // a multiple of 16
        if (valid >= 16) reinterpret_cast<uint4 *>(o)[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        if (valid >= 32) reinterpret_cast<uint4 *>(o)[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    } else {
        const int mw = (p.M + 31) >> 5, word = mc >> 5;
#pragma unroll
        for (int b = 0; b < OUT_BITS; ++b) {
            uint32_t bits = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) bits |= nibble_of_plane(packed[k], b) << (4 * k);
            reinterpret_cast<uint32_t *>(p.out)[((size_t)b * p.N + n) * mw + word] = bits;
        }
    }
}

}  // namespace qnn
