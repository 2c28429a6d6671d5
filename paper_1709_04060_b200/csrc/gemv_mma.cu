// Few-column GEMM (N <= 16) fused with the threshold activation, for every weight format: the fully
// connected layer at small batch of Section 4.2, whose gain the paper attributes to the packed
// weights' cut in memory traffic.  The weights are streamed once, in the form they are packed in,
// straight into registers, widened there to 8-bit values and multiplied by warp-level tensor-core
// instructions (mma.sync m16n8k32, int8 x int8 -> int32: exact, so the result is the integer that the
// bit-serial sum of Section 3.1 equals); T(x, t) of Section 2.1.1 is applied before anything is stored.
//
// Up to eight columns, sixteen weight rows are the instruction's first operand and the columns its second;
// beyond, the columns are the first and eight weight rows the second.  A warp owns a slice of the depth for
// all of its CTA's rows, so its part of the activations is loaded once, in the lane layout of the
// instruction, and stays in registers (up to 64 a lane): no shared memory, no barrier and nothing else than
// the weights' own loads between the start and the last row.  Rows are dealt in groups of eight, 8192 to 148
// SMs as 7 groups each (99 % even); a group is one byte of a bit-plane row.  A depth that the registers of
// 16 warps do not hold is walked in passes; a shallow one leaves warps over, which take other groups.
// Partial sums of all groups meet in shared memory once, at the end.
//
// Any order of the depth gives the same sum, so weights and activations only have to agree on one:
//   planes   a lane's word gives 32 elements, eight registers in the order of expand_word; the
//            activation words are widened by the same function
//   fields   a word masked at field position s holds four consecutive depth elements
//   bytes    a word is four elements as it stands
// A field that a mask leaves in the upper half of its byte pair is not shifted down: it counts 2^F times
// and has accumulators of its own, which are shifted back (exactly) when a group ends.  That leaves one
// AND a register with 4-bit fields and 1.25 to 1.4 instructions otherwise.
//
// Weights enter as unsigned offsets from the encoding's minimum (a bipolar one as its bit); the column
// sums of the activations, one more product with a column of ones, correct for the offset.
//
// What bounds it: two columns or so the weights (8192 x 8192 W2, 16.8 MB, 7.0 us; a plain read of as many bytes
// call after call takes 3.0 from L2 and more from HBM); 16 columns of bytes the activations, which every SM
// reads whole (131 KB each, 19 MB from L2).  8192 x 8192, us, activations staged through shared memory by the
// whole CTA -> here: planes W2A2 N = 2 8.4 -> 7.0, 4 9.1 -> 7.2, 16 14.8 -> 9.1, W4A4 N = 1 13.5 -> 11.5;
// fields W2 N = 2 7.8 -> 7.2, 16 12.3 -> 10.1, W4 N = 16 13.1 -> 11.9; bytes 1000 x 4096 N = 7 5.2 -> 3.3.
//
// 512 threads leave 128 registers a thread; of the 90 kernels the 29 with all 64 activation registers spill, 4 to 104
// bytes each (planes W1 word by word most, bytes 52, W2 fields 40 to 60, W4 fields 4 to 20).
#include "common.cuh"
#include "planes.cuh"

namespace qnn {

constexpr int MV_WARPS = 16, MV_THREADS = 32 * MV_WARPS;
constexpr int MV_COLS = 16;             // most columns
constexpr size_t MV_SMEM_MAX = SMEM_LIMIT;

enum { MV_PLANES = 0, MV_FIELDS = 1, MV_BYTES = 2 };

struct MvParams {
    const uint8_t *W, *A;
    const int32_t *thr;    // [M][n_thr] or null
    void *out;
    int M, N, K;
    int groups, per;       // groups of eight weight rows, in all and per CTA
    int units;             // loads (of V words) per weight row and plane
    int dsplit, rsplit;    // warps that share a row's depth; products that a CTA works on at a time
    int passes;            // parts of the depth, each held in registers as a whole
    long long w_pitch;     // bytes between weight rows
    long long w_plane;     // bytes between weight planes
    int a_bits, a_kind;    // planes: activation planes, PL_* kind
    int a_pitch;           // bytes between activation rows (planes: of one plane)
    int w_scale, w_off;
    uint32_t w_flip;       // planes: flips the top plane of a signed weight (offset binary)
    int out_bits, out_fmt, ld_out;
};

template <bool W_SIGNED, bool A_SIGNED>
__device__ __forceinline__ void mv_mma(int (&d)[4], uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, const uint32_t (&a)[2]) {
#define QNN_MV_MMA(WT_, AT_)                                                                                              \
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32." WT_ "." AT_ ".s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};" \
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(w0), "r"(w1), "r"(w2), "r"(w3), "r"(a[0]), "r"(a[1]))
    if (W_SIGNED && A_SIGNED) QNN_MV_MMA("s8", "s8");
    else if (W_SIGNED) QNN_MV_MMA("s8", "u8");
    else if (A_SIGNED) QNN_MV_MMA("u8", "s8");
    else QNN_MV_MMA("u8", "u8");
#undef QNN_MV_MMA
}
// The same with the activations as the 16-row operand (two blocks of columns) and eight weight rows.
template <bool W_SIGNED, bool A_SIGNED>
__device__ __forceinline__ void mv_mma16(int (&d)[4], const uint32_t (&a)[4], uint32_t w0, uint32_t w1) {
#define QNN_MV_MMA(WT_, AT_)                                                                                              \
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32." AT_ "." WT_ ".s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};" \
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(w0), "r"(w1))
    if (W_SIGNED && A_SIGNED) QNN_MV_MMA("s8", "s8");
    else if (W_SIGNED) QNN_MV_MMA("s8", "u8");
    else if (A_SIGNED) QNN_MV_MMA("u8", "s8");
    else QNN_MV_MMA("u8", "u8");
#undef QNN_MV_MMA
}

// V words of global memory.  volatile: the loads stay where they are written, all of a warp's first ones
// ahead of everything that waits for one of them.  Whole 16-byte units of weights are streamed (nothing
// reads them again); smaller ones leave the rest of their sector to the warp's next load.  Not .nc: the
// kernel is resident while the one ahead may still write the activations.
template <int V, bool STREAM>
__device__ __forceinline__ void mv_load(uint32_t *w, const uint8_t *p) {
    if (V == 4 && STREAM)
        asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1 % V]), "=r"(w[2 % V]), "=r"(w[3 % V]) : "l"(p));
    else if (V == 4)
        asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1 % V]), "=r"(w[2 % V]), "=r"(w[3 % V]) : "l"(p));
    else if (V == 2)
        asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1 % V]) : "l"(p));
    else
        asm volatile("ld.global.u32 %0, [%1];" : "=r"(w[0]) : "l"(p));
}

// A word of every plane of a weight row -> eight registers of four bytes, in pairs: pair k holds the
// elements that registers mv_slot(k) and mv_slot(k) + mv_next of expand_word hold, times 2^F for the odd
// pairs (F: 1, 2, 4 for 1, 2 and 3-4 planes).
template <int B> constexpr int mv_field = B == 1 ? 1 : (B == 2 ? 2 : 4);
template <int B> constexpr int mv_next = B == 1 ? 2 : 1;
template <int B> __host__ __device__ constexpr int mv_slot(int k) {
    return B == 1 ? (k & 1) + 4 * (k >> 1) : (B == 2 ? 2 * (k & 1) + 4 * (k >> 1) : 4 * (k & 1) + 2 * (k >> 1));
}
template <int B>
__device__ __forceinline__ void mv_expand(const uint32_t *w, uint32_t (&o)[4][2]) {
    if (B == 1) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < 2; ++i) o[k][i] = (w[0] >> (4 * (k >> 1) + 2 * i)) & (k & 1 ? 0x02020202u : 0x01010101u);
        return;
    }
    const uint32_t e[2] = {(w[0] & 0x55555555u) | ((w[1] << 1) & 0xAAAAAAAAu), ((w[0] >> 1) & 0x55555555u) | (w[1] & 0xAAAAAAAAu)};
    if (B == 2) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < 2; ++i) o[k][i] = (e[i] >> (4 * (k >> 1))) & (k & 1 ? 0x0C0C0C0Cu : 0x03030303u);
        return;
    }
    const uint32_t w3 = B == 4 ? w[3] : 0u;
    const uint32_t f[2] = {(w[2] & 0x55555555u) | ((w3 << 1) & 0xAAAAAAAAu), ((w[2] >> 1) & 0x55555555u) | (w3 & 0xAAAAAAAAu)};
    const uint32_t x[4] = {(e[0] & 0x33333333u) | ((f[0] << 2) & 0xCCCCCCCCu), (e[1] & 0x33333333u) | ((f[1] << 2) & 0xCCCCCCCCu),
                           ((e[0] >> 2) & 0x33333333u) | (f[0] & 0xCCCCCCCCu), ((e[1] >> 2) & 0x33333333u) | (f[1] & 0xCCCCCCCCu)};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int i = 0; i < 2; ++i) o[k][i] = x[2 * (k >> 1) + i] & (k & 1 ? 0xF0F0F0F0u : 0x0F0F0F0Fu);
}

// Steps of a buffer: the largest power of two up to `most` that divides the steps of a product.
__host__ __device__ constexpr int mv_buffer_steps(int most, int steps) { return most > steps || steps % most != 0 ? mv_buffer_steps(most / 2, steps) : most; }

// Activation registers of a product: for each half of its depth, the column g and (NT == 2) g + 8.
#define MV_AT(HALF_, BLOCK_) ((HALF_) * NT + (BLOCK_))
// Ints between the rows of a group's partial sums: two blocks of columns are stored column by column.
__host__ __device__ constexpr int mv_part_pitch(int nt) { return nt == 2 ? 20 : 8; }

// SRC: MV_*; B: weight planes, or bits per field; V: words per load; NT: blocks of eight columns; U: steps
// of a warp per product and pass.  A step is what the four lanes of a row load at once: 4 V words of every
// plane, or 64 bytes.
template <int SRC, int B, int V, int NT, int U, bool W_SIGNED, bool A_SIGNED>
__global__ void __launch_bounds__(MV_THREADS, 1)
gemv_mma_kernel(const MvParams p) {
    constexpr int PL = SRC == MV_PLANES ? B : 1;                   // loads per row and step
    constexpr int S = SRC == MV_FIELDS ? 8 / B : 1;                // field positions of a byte
    constexpr int RP = SRC == MV_PLANES ? 4 : 1;                   // activation planes as loaded
    constexpr int AP = SRC == MV_PLANES ? 4 * V : 2 * S;           // products per step
    constexpr int G = 3 - NT;                                      // groups per product: 16 weight rows, or 8 against 16 columns
    constexpr int PITCH = mv_part_pitch(NT);
    // two buffers of up to 16 registers a lane: steps per buffer, of one product's groups or of several
    // (of few: a launch that runs a product or two per warp waits for every line of code it fetches, also of
    // the products it skips)
    constexpr int FIT = 16 / (G * PL * V), STEPS = FIT >= 8 ? 8 : (FIT >= 4 ? 4 : (FIT >= 2 ? 2 : 1)), MOST = AP >= 8 ? 2 : 4;
    constexpr int UB = mv_buffer_steps(STEPS, U), Q = U > UB ? 1 : (STEPS / UB < MOST ? STEPS / UB : MOST), NB = U / UB;
    constexpr int TURN = NB == 1 ? 2 : (NB % 2 ? 2 * NB : NB);     // buffers per turn of the loop (even)
    constexpr int FIELD = SRC == MV_PLANES ? mv_field<B> : (SRC == MV_FIELDS ? B : 0);
    extern __shared__ __align__(16) uint8_t mv_smem[];
    int *part = reinterpret_cast<int *>(mv_smem);                  // [group][depth slice][8 rows][PITCH: 8 NT columns]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int d = warp % p.dsplit, r0 = warp / p.dsplit;
    const int g0 = blockIdx.x * p.per, ng = min(p.per, p.groups - g0);
    const int n_thr = p.thr ? (1 << p.out_bits) - 1 : 0;
    int *thr_s = part + (size_t)p.per * p.dsplit * 8 * PITCH;
    pdl_wait();
    pdl_trigger();

    // thresholds of the CTA's rows, on their way while the weights stream
    if (p.thr) {
        const int32_t *first = p.thr + (size_t)g0 * 8 * n_thr;
        const int count = min(ng * 8, p.M - g0 * 8) * n_thr;
        for (int i = threadIdx.x; i < count; i += (int)blockDim.x)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(thr_s + i)), "l"(first + i) : "memory");
    }

    uint32_t w[2][Q][UB][G][PL][V];
    // (warps past the plan's only help with the outputs)
    for (int pass = r0 < p.rsplit ? 0 : p.passes; pass < p.passes; ++pass) {
        const int unit0 = (pass * p.dsplit + d) * 4 * U + t;       // this lane's first load in a row
        // steps nb UB .. of the products of ordinal gi .. gi + Q - 1 among this warp's.  No predicates: rows past
        // the last one repeat it (their sums go nowhere), and loads past a row's end its last load (they meet
        // activations that are zero).
        auto load = [&](uint32_t (&x)[Q][UB][G][PL][V], int gi, int nb) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int prod = r0 + (gi + q) * p.rsplit, m = (g0 + G * prod) * 8 + g;
                if (G * prod >= ng) continue;                      // uniform
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    const uint8_t *row = p.W + (size_t)min(m + 8 * i, p.M - 1) * p.w_pitch;
#pragma unroll
                    for (int u = 0; u < UB; ++u) {
                        const uint8_t *at = row + (uint32_t)min(unit0 + 4 * (nb * UB + u), p.units - 1) * (4u * V);
#pragma unroll
                        for (int b = 0; b < PL; ++b) mv_load<V, true>(x[q][u][i][b], at + (size_t)b * p.w_plane);
                    }
                }
            }
        };

        // Weights that come from HBM go ahead of the activations, which all SMs read from L2 (fields, 8192 x 8192
        // W2, N = 16: 13.2 -> 11.9 us; bytes, N = 8 13.1 -> 12.1); planes are few activation bytes, and their
        // widening would have to wait for the weights
        if (SRC != MV_PLANES) {
            load(w[0], 0, 0);
            load(w[1], NB == 1 ? Q : 0, NB == 1 ? 0 : 1);
        }
        // ---- this warp's slice of the activations, columns g and g + 8: as they lie in memory ...
        uint32_t act[U][AP][2 * NT], raw[NT][U][RP][V];
#pragma unroll
        for (int h = 0; h < NT; ++h) {
            const int n = g + 8 * h;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int unit = unit0 + 4 * u;
                const bool in = n < p.N && unit < p.units;
                if (SRC == MV_PLANES) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
#pragma unroll
                        for (int v = 0; v < V; ++v) raw[h][u][b % RP][v] = 0u;
                        if (in && b < p.a_bits)
                            mv_load<V, false>(raw[h][u][b % RP], p.A + ((size_t)b * p.N + n) * p.a_pitch + (size_t)unit * (4 * V));
                    }
                } else if (SRC == MV_FIELDS && S >= 4) {
                    // The four lanes' 4 S pieces of 16 elements lie one behind the other: lanes 0 and 1 meet the
                    // even and odd ones of the first half, 2 and 3 of the second.  Loaded four neighbours at a time
                    // (as many lines as columns, not twice that: 8192 x 8192 N = 16, W2 12.3 -> 10.1 us, W1 10.7 -> 8.8),
                    // then half of them change places with lane t ^ 2.
                    uint32_t y[S][4];
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        const int au = (unit - t) * S + 4 * s + t;
#pragma unroll
                        for (int v = 0; v < 4; ++v) y[s][v] = 0u;
                        if (n < p.N && 16 * au < p.a_pitch) mv_load<4, false>(y[s], p.A + (size_t)n * p.a_pitch + 16 * (size_t)au);
                    }
#pragma unroll
                    for (int s = 0; s < S / 2; ++s)
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const uint32_t lo = y[s][v], hi = y[(s + S / 2) % S][v], got = __shfl_xor_sync(0xffffffffu, t < 2 ? hi : lo, 2);
                            act[u][(4 * s + (v >> 1)) % AP][MV_AT(v & 1, h)] = t < 2 ? lo : got;
                            act[u][(4 * s + 2 + (v >> 1)) % AP][MV_AT(v & 1, h)] = t < 2 ? got : hi;
                        }
                } else {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        // fields: half (unit & 1) of 32-byte group unit / 2 meets S pieces of 16 elements
                        const int au = SRC == MV_FIELDS ? (unit >> 1) * (2 * S) + 2 * s + (unit & 1) : unit;
                        uint32_t y[4] = {0u, 0u, 0u, 0u};
                        if (in && 16 * au < p.a_pitch) mv_load<4, false>(y, p.A + (size_t)n * p.a_pitch + 16 * (size_t)au);
#pragma unroll
                        for (int v = 0; v < 4; ++v) act[u][(2 * s + (v >> 1)) % AP][MV_AT(v & 1, h)] = y[v];
                    }
                }
            }
        }
        if (SRC == MV_PLANES) {
            load(w[0], 0, 0);
            load(w[1], NB == 1 ? Q : 0, NB == 1 ? 0 : 1);
        }
        // ... and planes widened, in the pairs mv_expand forms
        if (SRC == MV_PLANES) {
            auto words = [&](auto &&f) {
#pragma unroll
                for (int h = 0; h < NT; ++h)
#pragma unroll
                    for (int u = 0; u < U; ++u)
#pragma unroll
                        for (int v = 0; v < V; ++v) f(h, u, v);
            };
            if (p.a_bits <= 2)
                words([&](int h, int u, int v) {
                    const uint32_t a[4] = {raw[h][u][0][v], raw[h][u][1 % RP][v], 0u, 0u};
                    uint32_t o[8];
                    expand_word<2, PL_UNSIGNED>(a, o);             // planes past a_bits are zero
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        act[u][(4 * v + k) % AP][MV_AT(0, h)] = o[mv_slot<B>(k)];
                        act[u][(4 * v + k) % AP][MV_AT(1, h)] = o[mv_slot<B>(k) + mv_next<B>];
                    }
                });
            else
                words([&](int h, int u, int v) {
                    uint32_t a[4], o[8];
#pragma unroll
                    for (int b = 0; b < 4; ++b) a[b] = raw[h][u][b % RP][v];
                    expand_word<4, PL_UNSIGNED>(a, o);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        act[u][(4 * v + k) % AP][MV_AT(0, h)] = o[mv_slot<B>(k)];
                        act[u][(4 * v + k) % AP][MV_AT(1, h)] = o[mv_slot<B>(k) + mv_next<B>];
                    }
                });
            if (p.a_kind == PL_SIGNED) {
                // two's complement: the lower planes less the top one
                const uint32_t top = 0x01010101u << (p.a_bits - 1);
                words([&](int h, int u, int v) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        uint32_t &x = act[u][(4 * v + (k >> 1)) % AP][MV_AT(k & 1, h)];
                        x = (((x & ~top) | 0x80808080u) - (x & top)) ^ 0x80808080u;
                    }
                });
            } else if (p.a_kind == PL_BIPOLAR) {
                // +-1 has no zero: nothing past the depth, and nothing in an absent column
                words([&](int h, int u, int v) {
                    const int left = g + 8 * h < p.N ? p.K - 32 * ((unit0 + 4 * u) * V + v) : 0;
                    const uint32_t keep = left >= 32 ? 0xFFFFFFFFu : (left <= 0 ? 0u : (1u << left) - 1u);
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        uint32_t &x = act[u][(4 * v + (k >> 1)) % AP][MV_AT(k & 1, h)];
                        x = ((2u * x | 0x80808080u) - 0x01010101u) ^ 0x80808080u;
                        x &= ((keep >> (mv_slot<B>(k >> 1) + (k & 1) * mv_next<B>)) & 0x01010101u) * 0xFFu;
                    }
                });
            }
        }
        int cs[4] = {0, 0, 0, 0};                                  // column sums, in the layout of the accumulators
        if (p.w_off != 0) {
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int j = 0; j < AP; ++j) {
                    if constexpr (NT == 2) mv_mma16<false, A_SIGNED>(cs, act[u][j], 0x01010101u, 0x01010101u);
                    else mv_mma<false, A_SIGNED>(cs, 0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u, act[u][j]);
                }
#pragma unroll
            for (int e = 0; e < 4; ++e) cs[e] *= p.w_off;
        }

        int acc[2][4];                                             // even and odd pairs of registers
        auto multiply = [&](const uint32_t (&x)[Q][UB][G][PL][V], int gi, int nb) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const int prod = r0 + (gi + q) * p.rsplit;
                if (G * prod >= ng) continue;                      // uniform
                if (nb == 0) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[0][e] = acc[1][e] = 0;
                }
#pragma unroll
                for (int ub = 0; ub < UB; ++ub) {
                    const int u = nb * UB + ub;
                    if (SRC == MV_PLANES) {
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            uint32_t o[G][4][2];
#pragma unroll
                            for (int i = 0; i < G; ++i) {
                                uint32_t ww[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                                for (int b = 0; b < PL; ++b) ww[b] = b == PL - 1 ? x[q][ub][i][b][v] ^ p.w_flip : x[q][ub][i][b][v];
                                mv_expand<B>(ww, o[i]);
                            }
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if constexpr (NT == 2) mv_mma16<false, true>(acc[k & 1], act[u][(4 * v + k) % AP], o[0][k][0], o[0][k][1]);
                                else mv_mma<false, true>(acc[k & 1], o[0][k][0], o[G - 1][k][0], o[0][k][1], o[G - 1][k][1], act[u][(4 * v + k) % AP]);
                            }
                        }
                    } else {
                        constexpr uint32_t MASK = B == 1 ? 0x01010101u : (B == 2 ? 0x03030303u : (B == 4 ? 0x0F0F0F0Fu : 0xFFFFFFFFu));
#pragma unroll
                        for (int s = 0; s < S; ++s) {
                            uint32_t o[G][4];
#pragma unroll
                            for (int i = 0; i < G; ++i)
#pragma unroll
                                for (int v = 0; v < 4; ++v)
                                    o[i][v] = SRC == MV_FIELDS ? (x[q][ub][i][0][v % V] >> (B * (s & ~1))) & (MASK << (B * (s & 1))) : x[q][ub][i][0][v % V];
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                int (&a)[4] = acc[SRC == MV_FIELDS ? s & 1 : k];
                                if constexpr (NT == 2) mv_mma16<W_SIGNED, A_SIGNED>(a, act[u][(2 * s + k) % AP], o[0][2 * k], o[0][2 * k + 1]);
                                else mv_mma<W_SIGNED, A_SIGNED>(a, o[0][2 * k], o[G - 1][2 * k], o[0][2 * k + 1], o[G - 1][2 * k + 1], act[u][(2 * s + k) % AP]);
                            }
                        }
                    }
                }
                if (nb == NB - 1) {
                    int y[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) y[e] = p.w_scale * (acc[0][e] + (acc[1][e] >> FIELD)) + cs[e];
                    int *dst = part + (((size_t)(G * prod) * p.dsplit + d) * 8 + (NT == 2 ? 2 * t : g)) * PITCH + (NT == 2 ? g : 2 * t);
                    if constexpr (NT == 2) {
                        // rows 2 t and 2 t + 1, columns g and g + 8
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            int *q1 = dst + (e & 1) * PITCH + (e >> 1) * 8;
                            *q1 = pass > 0 ? *q1 + y[e] : y[e];
                        }
                    } else {
                        // rows g of two groups, columns 2 t and 2 t + 1
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            if (2 * prod + i >= ng) continue;
                            int2 *q1 = reinterpret_cast<int2 *>(dst + i * p.dsplit * 8 * PITCH);
                            int2 o = make_int2(y[2 * i], y[2 * i + 1]);
                            if (pass > 0) { const int2 a = *q1; o.x += a.x; o.y += a.y; }
                            *q1 = o;
                        }
                    }
                }
            }
        };
        for (int gi = 0; G * (r0 + gi * p.rsplit) < ng; gi += NB == 1 ? 2 * Q : TURN / NB) {
#pragma unroll
            for (int i = 0; i < TURN; ++i) {
                multiply(w[i & 1], NB == 1 ? gi + i * Q : gi + i / NB, NB == 1 ? 0 : i % NB);
                if (NB == 1) load(w[i & 1], gi + (i + 2) * Q, 0);
                else load(w[i & 1], gi + (i + 2) / NB, (i + 2) % NB);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // ---- all partial sums of an output, its thresholds, its code; eight lanes are the rows of a group
    const int total = ng * 8 * p.N;
    for (int base = warp * 32; base < total; base += (int)blockDim.x) {
        const int i = base + lane, row = i & 7, gn = (i >> 3) / p.N, gl = min(gn, ng - 1), n = (i >> 3) - gn * p.N;
        const int m = (g0 + gl) * 8 + row;
        const bool ok = i < total;
        const int *src = part + ((size_t)gl * p.dsplit * 8 + row) * PITCH + n;
        int x = 0;
#pragma unroll 8
        for (int v = 0; v < p.dsplit; ++v) x += src[v * 8 * PITCH];
        if (!p.thr) {
            if (ok && m < p.M) reinterpret_cast<int32_t *>(p.out)[(size_t)n * p.M + m] = x;
            continue;
        }
        int code = 0;
        if (m < p.M)
            for (int q = 0; q < n_thr; ++q) code += x >= thr_s[(gl * 8 + row) * n_thr + q] ? 1 : 0;
        if (p.out_fmt == QNN_FMT_INT8) {
            if (ok && m < p.ld_out) reinterpret_cast<uint8_t *>(p.out)[(size_t)n * p.ld_out + m] = (uint8_t)code;
        } else {
            // a group is one byte of the row's words
            const int mw = (p.M + 31) >> 5;
            for (int b = 0; b < p.out_bits; ++b) {
                const uint32_t bits = __ballot_sync(0xffffffffu, (code >> b) & 1) >> (lane & 24);
                if (ok && row == 0) reinterpret_cast<uint8_t *>(p.out)[((size_t)b * p.N + n) * 4 * mw + g0 + gl] = (uint8_t)bits;
            }
        }
    }
}

// ------------------------------------------------------------------- host side
struct MvPlan { int src, b, v, units, u, dsplit, rsplit, passes, groups, per, threads; size_t smem; };

// Activation registers per lane and step, and the steps of a warp per product that kernels are built for:
// as many as 64 such registers allow, three quarters of that (depths that leave warps idle otherwise), and fewer for
// shallow depths and few rows.
static int mv_act_regs(const MvPlan &pl, int nt) { return nt * (pl.src == MV_PLANES ? 8 * pl.v : 4 * (8 / pl.b)); }
constexpr int mv_steps_least(int regs) { return regs >= 16 ? 1 : (regs == 8 ? 2 : 4); }
constexpr int mv_steps_most(int regs) { return 64 / regs; }
constexpr int mv_steps_mid(int regs) { return mv_steps_most(regs) >= 4 ? mv_steps_most(regs) * 3 / 4 : mv_steps_most(regs); }

static bool mv_plan(const qnn_gemm_desc *d, bool has_thr, MvPlan *pl) {
    if (d->N > MV_COLS) return false;
    const int nt = d->N > 8 ? 2 : 1, sms = sm_count();
    if (d->w_fmt == QNN_FMT_BITPLANES) {
        if (d->w_bits > 4 || d->a_bits > 4) return false;
        const int kw = ceil_div(d->K, 32);
        pl->src = MV_PLANES; pl->b = d->w_bits;
        // 16-byte loads where rows are whole units of them and two rows' planes fit the registers, else 8-byte
        // ones where they can be, else words
        pl->v = kw % 4 == 0 && d->w_bits <= 2 ? 4 : (kw % 2 == 0 ? 2 : 1);
        pl->units = kw / pl->v;
    } else if (d->w_fmt == QNN_FMT_FIELDS) {
        pl->src = MV_FIELDS; pl->b = d->w_bits == 1 ? 1 : (d->w_bits == 2 ? 2 : 4); pl->v = 4;
        pl->units = 2 * ceil_div(d->K, 32 * (8 / pl->b));
    } else {
        if (d->N > 8) return false;                                // the tiled tensor-core kernel
        pl->src = MV_BYTES; pl->b = 8; pl->v = 4;
        pl->units = round_up(d->K, 16) / 16;
    }
    // rows in whole groups, and in what the output pads its rows to
    pl->groups = ceil_div(d->M, 8);
    if (has_thr) pl->groups = d->out_fmt == QNN_FMT_BITPLANES ? 4 * ceil_div(d->M, 32) : 2 * ceil_div(d->M, 16);
    // depth and rows to warps: fewest steps for the warp with the most; a pass waits for its activations,
    // which takes about as long as five steps (fields, us, five or more passes of one step -> two of four, W4
    // 4101 x 9063 N = 11: 11.1 -> 10.2; three of one -> two of two, W2 6154 x 8805 N = 16: 10.8 -> 12.5)
    const int steps = ceil_div(pl->units, 4), regs = mv_act_regs(*pl, nt), most = mv_steps_most(regs);
    long long best = 0;
    // (three quarters of the steps only where a row's depth takes more than half of the warps: 3597 x 9725 bytes, N = 5,
    // ten of sixteen 10.1 -> 7.6; where the rows are shared between warps the other two are the better ones)
    for (int u : {mv_steps_least(regs), mv_steps_mid(regs), most}) {
        if (u == mv_steps_mid(regs) && u < most && 2 * ceil_div(steps, most) <= MV_WARPS) continue;
        const int passes = ceil_div(steps, MV_WARPS * u), ds = ceil_div(steps, u * passes), rs = MV_WARPS / ds;
        const int fit = (int)((MV_SMEM_MAX - 1024) / (ds * 32 * mv_part_pitch(nt) + 8 * 15 * 4));
        const int waves = ceil_div(pl->groups, sms * fit), per = ceil_div(pl->groups, sms * waves);
        const int prods = ceil_div(per, 3 - nt);
        const long long cost = (long long)waves * passes * (ceil_div(prods, rs) * u + 5);
        if (best != 0 && cost >= best) continue;
        best = cost;
        pl->u = u; pl->passes = passes; pl->dsplit = ds; pl->rsplit = rs < prods ? rs : prods; pl->per = per;
    }
    // ... and enough warps for the outputs
    const int outputs = pl->per * 8 * d->N, want = outputs < 256 ? round_up(outputs, 32) : 256;
    pl->threads = 32 * pl->dsplit * pl->rsplit > want ? 32 * pl->dsplit * pl->rsplit : want;
    pl->smem = (size_t)pl->per * (pl->dsplit * 32 * mv_part_pitch(nt) + 8 * 15 * 4);
    return true;
}

// Bit planes: whether this kernel beats the one that counts bits (gemv_planes.cu), by an estimate of both in
// microseconds.  That one costs a load latency per staged column and plane, one per depth step of a lane, its CTAs
// and its population counts; this one its fill and drain, the products of the warp with the most, the weights, the
// columns it widens and the partial sums it exchanges.  The terms' shares are a non-negative least-squares fit to
// 7623 random problems timed with both kernels (half of them with one column; up to 12000 x 9216, every width,
// encoding and output), replayed as a graph; call after call this kernel takes a little longer, hence the factor.
// Twelve plane pairs and more of 2^22 weights are never counted: the estimate is up to a fifth off there (8192 x
// 8192 W4A4, one column: 14.6 us counted, 11.5 here).  One column of fewer pairs always is: a call by itself is up to
// 7 % faster here, but in a chain the layers around it weigh more (fully connected layers of the AlexNet-shaped
// network at batch 1: 68.7 us here, 65.6 counted); and so is one column in several passes (2021 problems 6000 to
// 60000 deep: this kernel 1.25 times as long on average).  On average the choice costs 0.6 % (graph) and 0.9 %
// (calls) of the faster one's time with two columns and more, 6.6 % and 3.0 % with one; always this kernel 0.4 % and
// 1.6 %, with one column 10 % and 11 %; always counting 128 % and 98 %, with one column 11 % and 3.7 %.
static bool mv_planes_faster(const qnn_gemm_desc *d, bool has_thr) {
    if (d->N == 1 && d->w_bits * d->a_bits < 12) return false;
    if (d->w_bits * d->a_bits >= 12 && (long long)d->M * d->K >= (1ll << 22)) return true;
    MvPlan pl;
    if (!mv_plan(d, has_thr, &pl) || (d->N == 1 && pl.passes > 1)) return false;
    const int kw = ceil_div(d->K, 32), cols = d->N < 4 ? d->N : 4, pairs = d->w_bits * d->a_bits, nt = d->N > 8 ? 2 : 1;
    const double ctas = (double)ceil_div(d->M, 8) * ceil_div(d->N, 4), words = (double)d->M * kw;
    const double staged = d->w_enc == QNN_ENC_BIPOLAR && d->a_enc != QNN_ENC_BIPOLAR ? 0.43 : 0.285;   // with column sums
    const double counted = 1.42 + staged * d->a_bits * cols * ceil_div(kw, 256) +
                           (kw % 4 == 0 ? 0.616 * ceil_div(kw, 128) : 0.183 * ceil_div(kw, 32)) +
                           0.0113 * pairs * cols * ceil_div(kw, 32) + 2.38e-7 * words * pairs * d->N + (1.56e-3 + 2.4e-4 * cols) * ctas;
    const double waves = (double)ceil_div(ceil_div(pl.groups, pl.per), sm_count());
    const double rounds = waves * pl.passes * ceil_div(ceil_div(pl.per, 3 - nt), pl.rsplit) * pl.u;
    const double here = 2.60 + rounds * (0.172 + 0.0142 * pl.v * d->w_bits) + 1.04e-6 * words * d->w_bits +
                        1.74e-4 * d->N * kw * d->a_bits + (nt == 2 ? 0.2 : 0.0) + 1.3e-3 * pl.dsplit * pl.per * d->N +
                        2.0 * (waves * pl.passes - 1.0);
    return counted > 1.1 * here;
}

// Where this kernel is the faster one of those that take the format (8192 x 8192, us, the other -> this):
//   fields  two columns on: W2A2 N = 2 10.2 -> 7.2, N = 4 13.0 -> 7.3, N = 16 15.4 -> 9.5 (N = 1 6.0 -> 7.1)
//   planes  mv_planes_faster (W2A2 N = 4 12.9 -> 7.2, N = 16 38 -> 9.1; W4A4 N = 1 14.6 -> 11.5)
//   bytes   three columns on from 2^23 weights, four from 3 x 2^20: N = 4 26 -> 11.6, N = 8 35 -> 12.1 (N = 2
//           4805 x 5120 5.4 -> 6.2); 11841 x 512 N = 7 6.1 -> 2.9, 416 x 7424 N = 6 6.8 -> 4.0.  Below, where
//           either takes 2 to 3 us, a call of the host takes longer than both, and of this one longest
//           (320 x 1401 N = 7: 2.9 -> 2.5 replayed, 4.08 -> 4.16 call after call)
//   codes   fields and bytes whose kernels need a second launch that clears the output first (bit planes that
//           they set bit by bit; pad bytes that they do not write): the host's second launch decides, call
//           after call (fields N = 1 10.2 -> 8.1, bytes 4096 x 9216 N = 1 12.8 -> 11.4); bytes only below 2^26
//           elements (8192 x 8192: 16.1 there, 17 here)
// Deep products are walked in passes, up to the 209 KB of column bytes (elements, times columns) that fitted an SM's
// shared memory when the columns were staged there.  Past it the kernels that take over need 2 to 8 times as long
// (5 to 8 columns: planes 7.5; 9 to 16: planes 3.8, fields 2.2).
bool gemv_mma_takes(const qnn_gemm_desc *d, bool has_thr) {
    if (d->N > (d->w_fmt == QNN_FMT_INT8 ? 8 : MV_COLS)) return false;
    const long long size = (long long)d->M * d->K, column_bytes = (long long)d->N * round_up(d->K, 32);
    if (column_bytes > 209 * 1024) return false;
    if (d->w_fmt == QNN_FMT_BITPLANES) {
        if (d->w_bits > 4 || d->a_bits > 4) return false;
        return mv_planes_faster(d, has_thr);
    }
    const bool padded = has_thr && (d->out_fmt == QNN_FMT_BITPLANES || (d->w_fmt != QNN_FMT_FIELDS && d->M % 16 != 0));
    if (d->w_fmt == QNN_FMT_FIELDS) return d->N >= 2 || padded;
    return (d->N >= 3 && size >= (1ll << 23)) || (d->N >= 4 && size >= (3ll << 20)) || (padded && size < (1ll << 26));
}

template <int SRC, int B, int V, int NT, int U, bool W_SIGNED, bool A_SIGNED>
static qnn_status mv_launch(const MvParams &p, const MvPlan &pl, cudaStream_t s) {
    auto kern = gemv_mma_kernel<SRC, B, V, NT, U, W_SIGNED, A_SIGNED>;
    static std::atomic<bool> attr_done[QNN_MAX_DEVICES];           // per instantiation and device
    const int dev = current_device();
    if (dev < 0 || !allow_smem(kern, MV_SMEM_MAX, attr_done[dev])) return QNN_ERR_CUDA;
    // programmatic dependent launch: a CTA has most of an SM's registers to itself, so early placement cannot
    // crowd several onto one SM; nothing is read before griddepcontrol.wait
    if (launch_pdl<MvParams>(kern, dim3((unsigned)ceil_div(p.groups, p.per)), pl.threads, pl.smem, s, p) != cudaSuccess) return QNN_ERR_CUDA;
    count_launch();
    return launch_status();
}

template <int SRC, int B, int V, int NT, bool W_SIGNED, bool A_SIGNED>
static qnn_status mv_launch_u(const MvParams &p, const MvPlan &pl, cudaStream_t s) {
    constexpr int REGS = NT * (SRC == MV_PLANES ? 8 * V : 4 * (8 / B)), LEAST = mv_steps_least(REGS), MID = mv_steps_mid(REGS), MOST = mv_steps_most(REGS);
    if (pl.u == LEAST) return mv_launch<SRC, B, V, NT, LEAST, W_SIGNED, A_SIGNED>(p, pl, s);
    if (pl.u == MID) return mv_launch<SRC, B, V, NT, MID, W_SIGNED, A_SIGNED>(p, pl, s);
    return mv_launch<SRC, B, V, NT, MOST, W_SIGNED, A_SIGNED>(p, pl, s);
}

template <int SRC, int B, int V, bool W_SIGNED, bool A_SIGNED>
static qnn_status mv_launch_n(const MvParams &p, const MvPlan &pl, cudaStream_t s) {
    if (SRC != MV_BYTES && p.N > 8) return mv_launch_u<SRC, B, V, SRC == MV_BYTES ? 1 : 2, W_SIGNED, A_SIGNED>(p, pl, s);
    return mv_launch_u<SRC, B, V, 1, W_SIGNED, A_SIGNED>(p, pl, s);
}

qnn_status gemv_mma_launch(const qnn_gemm_desc *d, const void *W, const void *A, const int32_t *thr, void *out, cudaStream_t s) {
    MvPlan pl;
    if (!mv_plan(d, thr != nullptr, &pl)) return QNN_ERR_UNSUPPORTED;
    MvParams p = {};
    p.W = (const uint8_t *)W; p.A = (const uint8_t *)A; p.thr = thr; p.out = out;
    p.M = d->M; p.N = d->N; p.K = d->K;
    p.groups = pl.groups; p.per = pl.per; p.units = pl.units;
    p.dsplit = pl.dsplit; p.rsplit = pl.rsplit; p.passes = pl.passes;
    p.a_bits = d->a_bits; p.a_kind = plane_kind(d->a_enc);
    p.a_pitch = pl.src == MV_PLANES ? 4 * ceil_div(d->K, 32) : round_up(d->K, 16);
    p.w_pitch = pl.src == MV_FIELDS ? 16ll * pl.units : p.a_pitch;
    p.w_plane = (long long)d->M * p.w_pitch;
    p.w_scale = 1;
    if (pl.src != MV_BYTES) {
        if (d->w_enc == QNN_ENC_BIPOLAR) { p.w_scale = 2; p.w_off = -1; }
        else if (d->w_enc == QNN_ENC_SIGNED) { p.w_off = -(1 << (d->w_bits - 1)); p.w_flip = 0xFFFFFFFFu; }
    }
    p.out_bits = thr ? d->out_bits : 0;
    p.out_fmt = d->out_fmt;
    p.ld_out = round_up(d->M, 16);
    const bool as = d->a_enc != QNN_ENC_UNSIGNED, ws = d->w_enc != QNN_ENC_UNSIGNED;
    if (pl.src == MV_BYTES) {
        if (ws) return as ? mv_launch_n<MV_BYTES, 8, 4, true, true>(p, pl, s) : mv_launch_n<MV_BYTES, 8, 4, true, false>(p, pl, s);
        return as ? mv_launch_n<MV_BYTES, 8, 4, false, true>(p, pl, s) : mv_launch_n<MV_BYTES, 8, 4, false, false>(p, pl, s);
    }
    if (pl.src == MV_FIELDS) {
#define QNN_MV_CASE(B_) if (pl.b == B_) return as ? mv_launch_n<MV_FIELDS, B_, 4, false, true>(p, pl, s) : mv_launch_n<MV_FIELDS, B_, 4, false, false>(p, pl, s);
        QNN_MV_CASE(1) QNN_MV_CASE(2) QNN_MV_CASE(4)
#undef QNN_MV_CASE
    }
    // planes: at most four, so the activations fit signed bytes whatever their encoding
#define QNN_MV_CASE(B_)                                                                                                        \
    if (pl.b == B_) return pl.v == 4 ? mv_launch_n<MV_PLANES, B_, B_ <= 2 ? 4 : 2, false, true>(p, pl, s)                       \
                                     : (pl.v == 2 ? mv_launch_n<MV_PLANES, B_, 2, false, true>(p, pl, s) : mv_launch_n<MV_PLANES, B_, 1, false, true>(p, pl, s));
    QNN_MV_CASE(1) QNN_MV_CASE(2) QNN_MV_CASE(3) QNN_MV_CASE(4)
#undef QNN_MV_CASE
    return QNN_ERR_UNSUPPORTED;
}

}  // namespace qnn
