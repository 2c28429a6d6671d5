// Few-column GEMM (N <= 16) fused with the threshold activation, for every weight format: the fully
// connected layer at small batch of Section 4.2, whose gain the paper attributes to the packed
// weights' cut in memory traffic.  The weights are streamed once, in the form they are packed in,
// straight into registers, widened there to 8-bit values and multiplied by warp-level tensor-core
// instructions (mma.sync m16n8k32, int8 x int8 -> int32: exact, so the result is the integer that the
// bit-serial sum of Section 3.1 equals); T(x, t) of Section 2.1.1 is applied before anything is stored.
//
// What bounds it: up to eight columns the weights' latency and the fill and drain of an SM (8192 x 8192
// W2A2 fields, 16.8 MB: 8.0 us for 2 to 4 columns, against 10 to 13 in the other forms; 2.5 us at the copy
// rate), beyond them also the int8 rate of mma.sync, which is no more than that of dp4a here (12.3 us
// at 16).  The per-lane operand layout lets a loaded word feed the multiplication without a trip
// through shared or tensor memory, so columns up to eight come at one price and an SM holds nothing but
// loads in flight (16 warps x 8 x 16 bytes per lane, twice); tcgen05 would need every widened byte
// written to shared or tensor memory first, and 128-row tiles.  Any order of the depth gives the same
// sum, so weights and activations only have to agree on one:
//   planes   a lane's word gives 32 elements, eight registers in the order of expand_word; the
//            activation words are widened once per CTA by the same function
//   fields   a word masked at field position s holds four consecutive depth elements
//   bytes    a word is four elements as it stands
// Weights enter as unsigned offsets from the encoding's minimum (a bipolar one as its bit); the column
// sums of the activations correct for the offset, as in the packed-fields kernels.
//
// CTA = 16 warps, one CTA per SM, tiles of 32 weight rows (one word of the bit-plane output layout); the
// warps split the depth of a tile, and meet in shared memory, where warp n finishes column n.  A
// warp has two buffers of loads in flight, across tiles too (one at the start: 0.4 us slower).  512
// threads leave 128 registers each: bytes spill 24 bytes, planes with two blocks of columns 4 to 44
// (one and two planes with four-word loads), fields none.
#include "common.cuh"
#include "planes.cuh"

namespace qnn {

constexpr int MV_WARPS = 16, MV_THREADS = 32 * MV_WARPS;
constexpr int MV_ROWS = 32;             // weight rows per tile
constexpr int MV_COLS = 16;             // most columns
constexpr int MV_PART_PITCH = 36;       // partial sums [column][row], row pitch without bank conflicts
constexpr size_t MV_SMEM_MAX = SMEM_LIMIT;

enum { MV_PLANES = 0, MV_FIELDS = 1, MV_BYTES = 2 };

struct MvParams {
    const uint8_t *W, *A;
    const int32_t *thr;    // [M][n_thr] or null
    void *out;
    int M, N, K;
    int tiles, steps;      // 32-row tiles; steps of the depth per row
    int units;             // loads (of V words) per weight row, per plane
    long long w_pitch;     // bytes between weight rows
    long long w_plane;     // bytes between weight planes
    int a_bits, a_kind;    // planes: activation planes, PL_* kind
    int a_pitch;           // bytes between activation rows (planes: of one plane)
    int col_pitch;         // shared-memory bytes between activation columns
    int a_signed, w_scale, w_off;
    uint32_t w_flip;       // planes: flips the top plane of a signed weight (offset binary)
    int out_bits, out_fmt, ld_out;
};

template <bool W_SIGNED, bool A_SIGNED>
__device__ __forceinline__ void mv_mma(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
#define QNN_MV_MMA(WT_, AT_)                                                                                              \
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32." WT_ "." AT_ ".s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};" \
                 : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1))
    if (W_SIGNED && A_SIGNED) QNN_MV_MMA("s8", "s8");
    else if (W_SIGNED) QNN_MV_MMA("s8", "u8");
    else if (A_SIGNED) QNN_MV_MMA("u8", "s8");
    else QNN_MV_MMA("u8", "u8");
#undef QNN_MV_MMA
}

__device__ __forceinline__ uint4 mv_lds(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}

// V words of streamed weights (not kept in L1: nothing reads them again).
template <int V>
__device__ __forceinline__ void mv_load(uint32_t *w, const uint8_t *p) {
    if (V == 4) {
        const uint4 x = __ldcs(reinterpret_cast<const uint4 *>(p));
        w[0] = x.x; w[1] = x.y; w[2] = x.z; w[3] = x.w;
    } else if (V == 2) {
        const uint2 x = __ldcs(reinterpret_cast<const uint2 *>(p));
        w[0] = x.x; w[1] = x.y;
    } else {
        w[0] = __ldcs(reinterpret_cast<const uint32_t *>(p));
    }
}

// Shared-memory offset of 16-byte unit u of an activation column (fields).  The four lanes of a row read
// both halves of two neighbouring groups of 32 S bytes: where a group is a whole number of bank rows
// (S = 4, 8) 32 pad bytes per group keep them apart.
template <int S>
__device__ __forceinline__ uint32_t mv_field_unit(uint32_t u) { return S == 2 ? 16u * u : 16u * u + 32u * (u / (2 * S)); }

// SRC: MV_*; B: weight planes, or bits per field; V: words per load; NT: blocks of eight columns.
// A step of the depth is what the four lanes of a row load at once: 4 V words of every plane, or 64
// bytes.  U steps are in flight per warp and buffer.
template <int SRC, int B, int V, int NT, bool W_SIGNED, bool A_SIGNED>
__global__ void __launch_bounds__(MV_THREADS, 1)
gemv_mma_kernel(const MvParams p) {
    constexpr int PL = SRC == MV_PLANES ? B : 1;                   // loads per row and step
    constexpr int U = 8 / (PL * V) > 0 ? 8 / (PL * V) : 1;
    constexpr int S = SRC == MV_FIELDS ? 8 / B : 1;
    extern __shared__ __align__(16) uint8_t mv_smem[];
    int *part = reinterpret_cast<int *>(mv_smem);                  // [warp][8 NT columns][MV_PART_PITCH]
    uint8_t *cols = mv_smem + MV_WARPS * 8 * NT * MV_PART_PITCH * 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    pdl_wait();
    pdl_trigger();

    // ---- the warp's work: steps warp, warp + 16, ... of every tile of this CTA, U at a time
    int ld_tile = blockIdx.x, ld_step = warp;
    uint32_t w[2][U][4][PL][V];
    auto load = [&](uint32_t (&x)[U][4][PL][V]) {
        const bool live = ld_tile < p.tiles;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int unit = (ld_step + u * MV_WARPS) * 4 + t;
            const bool in = live && unit < p.units;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int m = ld_tile * MV_ROWS + g + 8 * r;
                const uint8_t *q = p.W + (size_t)m * p.w_pitch + (size_t)unit * (4 * V);
#pragma unroll
                for (int b = 0; b < PL; ++b) {
                    if (in && m < p.M) {
                        mv_load<V>(x[u][r][b], q + (size_t)b * p.w_plane);
                    } else {
#pragma unroll
                        for (int v = 0; v < V; ++v) x[u][r][b][v] = 0u;
                    }
                }
            }
        }
        ld_step += U * MV_WARPS;
        if (ld_step - warp >= p.steps) { ld_step = warp; ld_tile += gridDim.x; }
    };
    load(w[0]);
    load(w[1]);

    // ---- activation columns into shared memory, in the order the multiplication reads them
    if (SRC == MV_PLANES) {
        // word c of a column: step c / 4V, lane (c mod 4V) / V, word c mod V of the lane; 32 bytes each,
        // the four lanes' words next to one another
        const int words = p.steps * 4 * V, kw = p.a_pitch >> 2;
        for (int i = threadIdx.x; i < p.N * words; i += MV_THREADS) {
            const int n = i / words, c = i - n * words;
            uint32_t a[4] = {0u, 0u, 0u, 0u}, o[8];
            if (c < kw)
                for (int b = 0; b < p.a_bits; ++b)
                    a[b] = reinterpret_cast<const uint32_t *>(p.A)[((size_t)b * p.N + n) * kw + c];
            if (p.a_kind == PL_BIPOLAR) {
                expand_word<1, PL_BIPOLAR>(a, o);
                const int left = p.K - 32 * c;                     // +-1 has no zero: nothing past the depth
                const uint32_t keep = left >= 32 ? 0xFFFFFFFFu : (left <= 0 ? 0u : (1u << left) - 1u);
#pragma unroll
                for (int j = 0; j < 8; ++j) o[j] &= ((keep >> j) & 0x01010101u) * 0xFFu;
            } else if (p.a_kind == PL_SIGNED) {
                switch (p.a_bits) {
                    case 1: expand_word<1, PL_SIGNED>(a, o); break;
                    case 2: expand_word<2, PL_SIGNED>(a, o); break;
                    case 3: expand_word<3, PL_SIGNED>(a, o); break;
                    default: expand_word<4, PL_SIGNED>(a, o); break;
                }
            } else {
                expand_word<4, PL_UNSIGNED>(a, o);                 // planes past a_bits are zero
            }
            const int step = c / (4 * V), in = c % (4 * V), slot = step * 4 * V + (in % V) * 4 + in / V;
            uint4 *dst = reinterpret_cast<uint4 *>(cols + (size_t)n * p.col_pitch + 32 * slot);
            dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
            dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
        }
    } else {
        // plain bytes; what lies past the row meets zero weights, but has to be there
        const int units = p.a_pitch >> 4;
        for (int i = threadIdx.x; i < p.N * units; i += MV_THREADS) {
            const int n = i / units, u = i - n * units;
            *reinterpret_cast<uint4 *>(cols + (size_t)n * p.col_pitch + (SRC == MV_FIELDS ? mv_field_unit<S>(u) : 16u * u)) =
                reinterpret_cast<const uint4 *>(p.A + (size_t)n * p.a_pitch)[u];
        }
    }
    __syncthreads();
    int colsum = 0;                                                // warp n: sum of column n
    if (p.w_off != 0 && warp < p.N) {
        const int units = SRC == MV_PLANES ? p.steps * 8 * V : p.a_pitch >> 4;
        for (int u = lane; u < units; u += 32) {
            const uint4 a = *reinterpret_cast<const uint4 *>(cols + (size_t)warp * p.col_pitch + (SRC == MV_FIELDS ? mv_field_unit<S>(u) : 16u * u));
            if (A_SIGNED) {
                colsum = __dp4a((int)a.x, 0x01010101, colsum); colsum = __dp4a((int)a.y, 0x01010101, colsum);
                colsum = __dp4a((int)a.z, 0x01010101, colsum); colsum = __dp4a((int)a.w, 0x01010101, colsum);
            } else {
                colsum = (int)__dp4a(a.x, 0x01010101u, (unsigned)colsum); colsum = (int)__dp4a(a.y, 0x01010101u, (unsigned)colsum);
                colsum = (int)__dp4a(a.z, 0x01010101u, (unsigned)colsum); colsum = (int)__dp4a(a.w, 0x01010101u, (unsigned)colsum);
            }
        }
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) colsum += __shfl_xor_sync(0xffffffffu, colsum, off);
    }

    // this lane's column of each block (columns past N read the last one; their sums are not used)
    uint32_t col_at[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
        col_at[nt] = (uint32_t)__cvta_generic_to_shared(cols) + (uint32_t)min(8 * nt + g, p.N - 1) * (uint32_t)p.col_pitch;

    const int n_thr = p.thr ? (1 << p.out_bits) - 1 : 0;
    int acc[2][NT][4];
    auto multiply = [&](const uint32_t (&x)[U][4][PL][V], int step0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int step = step0 + u * MV_WARPS;
            if (step < p.steps) {                                  // uniform
                if (SRC == MV_PLANES) {
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        uint32_t bq[NT][8];
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            const uint32_t at = col_at[nt] + 32u * (uint32_t)(step * 4 * V + v * 4 + t);
                            const uint4 lo = mv_lds(at), hi = mv_lds(at + 16u);
                            bq[nt][0] = lo.x; bq[nt][1] = lo.y; bq[nt][2] = lo.z; bq[nt][3] = lo.w;
                            bq[nt][4] = hi.x; bq[nt][5] = hi.y; bq[nt][6] = hi.z; bq[nt][7] = hi.w;
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t o0[8], o1[8], wa[4], wb[4];
#pragma unroll
                            for (int b = 0; b < PL; ++b) {
                                const uint32_t f = b == PL - 1 ? p.w_flip : 0u;
                                wa[b] = x[u][2 * h][b][v] ^ f; wb[b] = x[u][2 * h + 1][b][v] ^ f;
                            }
                            expand_word<PL, PL_UNSIGNED>(wa, o0);
                            expand_word<PL, PL_UNSIGNED>(wb, o1);
#pragma unroll
                            for (int j = 0; j < 4; ++j)
#pragma unroll
                                for (int nt = 0; nt < NT; ++nt)
                                    mv_mma<false, A_SIGNED>(acc[h][nt], o0[2 * j], o1[2 * j], o0[2 * j + 1], o1[2 * j + 1],
                                                            bq[nt][2 * j], bq[nt][2 * j + 1]);
                        }
                    }
                } else {
#pragma unroll
                    for (int s = 0; s < S; ++s) {
                        constexpr uint32_t MASK = B == 1 ? 0x01010101u : (B == 2 ? 0x03030303u : (B == 4 ? 0x0F0F0F0Fu : 0xFFFFFFFFu));
                        uint4 bq[NT];
#pragma unroll
                        for (int nt = 0; nt < NT; ++nt) {
                            // fields: lane t holds half t & 1 of 32-byte group 2 step + t / 2
                            const uint32_t unit = SRC == MV_FIELDS ? (uint32_t)((2 * step + (t >> 1)) * 2 * S + 2 * s + (t & 1)) : (uint32_t)(4 * step + t);
                            bq[nt] = mv_lds(col_at[nt] + (SRC == MV_FIELDS ? mv_field_unit<S>(unit) : 16u * unit));
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t o0[4], o1[4];
#pragma unroll
                            for (int v = 0; v < 4; ++v) {
                                o0[v] = SRC == MV_FIELDS ? (x[u][2 * h][0][v] >> (B * s)) & MASK : x[u][2 * h][0][v];
                                o1[v] = SRC == MV_FIELDS ? (x[u][2 * h + 1][0][v] >> (B * s)) & MASK : x[u][2 * h + 1][0][v];
                            }
#pragma unroll
                            for (int nt = 0; nt < NT; ++nt) {
                                mv_mma<W_SIGNED, A_SIGNED>(acc[h][nt], o0[0], o1[0], o0[1], o1[1], bq[nt].x, bq[nt].y);
                                mv_mma<W_SIGNED, A_SIGNED>(acc[h][nt], o0[2], o1[2], o0[3], o1[3], bq[nt].z, bq[nt].w);
                            }
                        }
                    }
                }
            }
        }
    };

    const int rounds = (p.steps + U * MV_WARPS - 1) / (U * MV_WARPS);      // buffers per tile
    int cur = 0;
    for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[h][nt][e] = 0;
        int step = warp;
        for (int r = 0; r < rounds; ++r, step += U * MV_WARPS) {
            if (cur == 0) { multiply(w[0], step); load(w[0]); }
            else { multiply(w[1], step); load(w[1]); }
            cur ^= 1;
        }
        // thresholds of this thread's row, on their way while the partial sums meet
        const int m = tile * MV_ROWS + lane;
        int th[15];
        if (warp < p.N) {
#pragma unroll
            for (int q = 0; q < 15; ++q) th[q] = q < n_thr && m < p.M ? __ldg(p.thr + (size_t)m * n_thr + q) : 0x7fffffff;
        }
        int *mine = part + warp * (8 * NT * MV_PART_PITCH);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    mine[(8 * nt + 2 * t + (e & 1)) * MV_PART_PITCH + 16 * h + g + 8 * (e >> 1)] = acc[h][nt][e];
        __syncthreads();
        if (warp < p.N) {
            const int n = warp;
            int x = 0;
#pragma unroll
            for (int v = 0; v < MV_WARPS; ++v) x += part[(v * 8 * NT + n) * MV_PART_PITCH + lane];
            x = p.w_scale * x + p.w_off * colsum;
            if (!p.thr) {
                if (m < p.M) reinterpret_cast<int32_t *>(p.out)[(size_t)n * p.M + m] = x;
            } else {
                int code = 0;
#pragma unroll
                for (int q = 0; q < 15; ++q) code += q < n_thr && x >= th[q] ? 1 : 0;
                if (m >= p.M) code = 0;
                if (p.out_fmt == QNN_FMT_INT8) {
                    if (m < p.ld_out) reinterpret_cast<uint8_t *>(p.out)[(size_t)n * p.ld_out + m] = (uint8_t)code;
                } else {
                    const int mw = (p.M + 31) >> 5;
                    for (int b = 0; b < p.out_bits; ++b) {
                        const uint32_t bits = __ballot_sync(0xffffffffu, (code >> b) & 1);
                        if (lane == 0) reinterpret_cast<uint32_t *>(p.out)[((size_t)b * p.N + n) * mw + tile] = bits;
                    }
                }
            }
        }
        __syncthreads();                                           // the partial sums have been read
    }
}

// ------------------------------------------------------------------- host side
struct MvPlan { int src, b, v, units, steps, col_pitch; size_t smem; };

static bool mv_plan(const qnn_gemm_desc *d, MvPlan *pl) {
    if (d->N > MV_COLS) return false;
    const int nt = d->N > 8 ? 2 : 1;
    long long col = 0;
    if (d->w_fmt == QNN_FMT_BITPLANES) {
        if (d->w_bits > 4 || d->a_bits > 4) return false;
        const int kw = ceil_div(d->K, 32);
        pl->src = MV_PLANES; pl->b = d->w_bits;
        // Wide loads once they leave every warp a step of its own (and with few planes: registers);
        // rows that are not whole units go word by word.
        pl->v = kw % 4 == 0 && kw >= 16 * MV_WARPS && d->w_bits <= 2 ? 4 : (kw % 2 == 0 && kw >= 8 * MV_WARPS ? 2 : 1);
        pl->units = kw / pl->v;
        pl->steps = ceil_div(pl->units, 4);
        col = 128ll * pl->steps * pl->v;
        pl->col_pitch = (int)(col + 16);                           // eight lanes (two columns) on different banks
    } else if (d->w_fmt == QNN_FMT_FIELDS) {
        const int f = d->w_bits == 1 ? 1 : (d->w_bits == 2 ? 2 : 4), S = 8 / f;
        const int ldf = 32 * ceil_div(d->K, 32 * S);
        pl->src = MV_FIELDS; pl->b = f; pl->v = 4;
        pl->units = ldf / 16;
        pl->steps = ceil_div(pl->units, 4);
        col = (long long)pl->steps * 2 * (32 * S + (S == 2 ? 0 : 32));
        pl->col_pitch = (int)(col + 127) / 128 * 128 + (S == 2 ? 32 : 64);   // two columns on different banks
    } else {
        if (d->N > 8) return false;                                // the tiled tensor-core kernel
        pl->src = MV_BYTES; pl->b = 8; pl->v = 4;
        pl->units = round_up(d->K, 16) / 16;
        pl->steps = ceil_div(pl->units, 4);
        col = (long long)pl->steps * 64;
        pl->col_pitch = (int)(col + 127) / 128 * 128 + 64;
    }
    if (col > (long long)MV_SMEM_MAX) return false;
    pl->smem = (size_t)MV_WARPS * 8 * nt * MV_PART_PITCH * 4 + (size_t)d->N * pl->col_pitch;
    return pl->smem <= MV_SMEM_MAX;
}

// Bit planes that need no clearing launch: whether this kernel beats the one that counts bits
// (gemv_planes.cu), by an estimate of both in microseconds.  That one costs a load latency per staged
// column and plane, one per depth step of a lane, its CTAs and its population counts; this one its fill
// and drain, the columns it widens, the rounds of tiles and the weights.  Fitted to 3300 random problems
// (1 to 16 columns, up to 12000 x 9216, every width and encoding, replayed as a graph): the choice costs
// 0.8 % of the faster one's time on average, always this kernel 14 % (959 x 64, N = 5, W2A1: 2.7 us there,
// 4.7 here), always the other 49 %.
static bool mv_planes_faster(const qnn_gemm_desc *d) {
    const int kw = ceil_div(d->K, 32), cols = d->N < 4 ? d->N : 4, pairs = d->w_bits * d->a_bits;
    const double ctas = (double)ceil_div(d->M, 8) * ceil_div(d->N, 4), words = (double)d->M * kw;
    const double staged = d->w_enc == QNN_ENC_BIPOLAR && d->a_enc != QNN_ENC_BIPOLAR ? 0.48 : 0.32;   // with column sums
    const double counted = 0.89 + staged * d->a_bits * cols * ceil_div(kw, 256) +
                           (kw % 4 == 0 ? 0.83 * ceil_div(kw, 128) : 0.23 * ceil_div(kw, 32)) +
                           0.011 * pairs * cols * ceil_div(kw, 32) + 2.3e-7 * words * pairs * d->N + 2.44e-3 * ctas;
    const double here = (d->w_bits <= 2 ? 4.8 : 4.0) + (d->N > 8 ? 0.25 : 0.0) + 1.9e-3 * d->N * kw +
                        1.5 * ((ceil_div(d->M, MV_ROWS) - 1) / sm_count()) + 0.8e-6 * words * d->w_bits;
    return counted > 0.96 * here;
}

// Where this kernel is the faster one of those that take the format (8192 x 8192, us, the other -> this):
//   fields  two columns on: W2A2 N = 2 10.2 -> 8.0, N = 4 13.0 -> 8.0, N = 16 15.4 -> 12.3 (N = 1 6.2 -> 7.8)
//   planes  two columns on, or one where there are twelve or more plane pairs to count (8192 x 8192, weights
//           in L2: W2A2 N = 4 12.9 -> 8.8, N = 16 38 -> 14.6, N = 2 the same; W4A4 N = 1 14.6 -> 13.1, from
//           HBM the same), but for small problems: mv_planes_faster
//   bytes   three columns on: N = 4 26 -> 17, N = 8 35 -> 18 (N = 2 15.9 -> 17.6), and not for small
//           matrices (1000 x 4096, N = 7: 4.6 -> 4.9)
//   any     where the others need a second launch that clears the output first (bit planes they set
//           bit by bit; pad bytes they do not write), the host's second launch decides, call after call
//           (planes: 4.6 us here, 7.3 there for everything small, and faster here for 677 of 700 random
//           problems up to 12000 x 9216, although one in five takes longer on the device, up to 3 us;
//           fields N = 1 10.2 -> 8.1, bytes 4096 x 9216 N = 1 12.8 -> 11.4); bytes only below 2^26
//           elements (8192 x 8192: 16.1 there, 17 here), planes with one column below 2^24 (from there on
//           the two launches take less time on the device: 66.9 against 67.6 us for the batch-1 chain as
//           a graph)
bool gemv_mma_takes(const qnn_gemm_desc *d, bool has_thr) {
    MvPlan pl;
    if (!mv_plan(d, &pl)) return false;
    const bool clears = has_thr && (d->out_fmt == QNN_FMT_BITPLANES || (pl.src != MV_FIELDS && d->M % 16 != 0));
    if (pl.src == MV_FIELDS) return d->N >= 2 || clears;
    const long long size = (long long)d->M * d->K;
    if (pl.src == MV_PLANES)
        return clears ? d->N >= 2 || d->w_bits * d->a_bits >= 12 || size < (1ll << 24)
                      : (d->N >= 2 || d->w_bits * d->a_bits >= 12) && mv_planes_faster(d);
    return (d->N >= 3 && size >= (1ll << 23)) || (clears && size < (1ll << 26));
}

template <int SRC, int B, int V, int NT, bool W_SIGNED, bool A_SIGNED>
static qnn_status mv_launch(const MvParams &p, size_t smem, cudaStream_t s) {
    auto kern = gemv_mma_kernel<SRC, B, V, NT, W_SIGNED, A_SIGNED>;
    static std::atomic<bool> attr_done[QNN_MAX_DEVICES];           // per instantiation and device
    const int dev = current_device();
    if (dev < 0 || !allow_smem(kern, MV_SMEM_MAX, attr_done[dev])) return QNN_ERR_CUDA;
    // programmatic dependent launch: a CTA has an SM's registers to itself, so early placement cannot
    // crowd several onto one SM; nothing is read before griddepcontrol.wait
    const dim3 grid((unsigned)(p.tiles < sm_count() ? p.tiles : sm_count()));
    if (launch_pdl<MvParams>(kern, grid, MV_THREADS, smem, s, p) != cudaSuccess) return QNN_ERR_CUDA;
    count_launch();
    return launch_status();
}

template <int SRC, int B, int V, bool W_SIGNED>
static qnn_status mv_launch_n(const MvParams &p, size_t smem, cudaStream_t s) {
    if (SRC != MV_BYTES && p.N > 8)
        return p.a_signed ? mv_launch<SRC, B, V, SRC == MV_BYTES ? 1 : 2, W_SIGNED, true>(p, smem, s)
                          : mv_launch<SRC, B, V, SRC == MV_BYTES ? 1 : 2, W_SIGNED, false>(p, smem, s);
    return p.a_signed ? mv_launch<SRC, B, V, 1, W_SIGNED, true>(p, smem, s) : mv_launch<SRC, B, V, 1, W_SIGNED, false>(p, smem, s);
}

qnn_status gemv_mma_launch(const qnn_gemm_desc *d, const void *W, const void *A, const int32_t *thr, void *out, cudaStream_t s) {
    MvPlan pl;
    if (!mv_plan(d, &pl)) return QNN_ERR_UNSUPPORTED;
    MvParams p = {};
    p.W = (const uint8_t *)W; p.A = (const uint8_t *)A; p.thr = thr; p.out = out;
    p.M = d->M; p.N = d->N; p.K = d->K;
    p.tiles = ceil_div(d->M, MV_ROWS); p.steps = pl.steps; p.units = pl.units;
    p.a_bits = d->a_bits; p.a_kind = plane_kind(d->a_enc);
    p.a_pitch = pl.src == MV_PLANES ? 4 * ceil_div(d->K, 32) : round_up(d->K, 16);
    p.w_pitch = pl.src == MV_FIELDS ? 16ll * pl.units : p.a_pitch;
    p.w_plane = (long long)d->M * p.w_pitch;
    p.col_pitch = pl.col_pitch;
    p.a_signed = d->a_enc != QNN_ENC_UNSIGNED ? 1 : 0;
    p.w_scale = 1;
    if (pl.src != MV_BYTES) {
        if (d->w_enc == QNN_ENC_BIPOLAR) { p.w_scale = 2; p.w_off = -1; }
        else if (d->w_enc == QNN_ENC_SIGNED) { p.w_off = -(1 << (d->w_bits - 1)); p.w_flip = 0xFFFFFFFFu; }
    }
    p.out_bits = thr ? d->out_bits : 0;
    p.out_fmt = d->out_fmt;
    p.ld_out = round_up(d->M, 16);
    const size_t m = pl.smem;
    if (pl.src == MV_BYTES)
        return d->w_enc != QNN_ENC_UNSIGNED ? mv_launch_n<MV_BYTES, 8, 4, true>(p, m, s) : mv_launch_n<MV_BYTES, 8, 4, false>(p, m, s);
    if (pl.src == MV_FIELDS)
        return pl.b == 1 ? mv_launch_n<MV_FIELDS, 1, 4, false>(p, m, s)
                         : (pl.b == 2 ? mv_launch_n<MV_FIELDS, 2, 4, false>(p, m, s) : mv_launch_n<MV_FIELDS, 4, 4, false>(p, m, s));
#define QNN_MV_CASE(B_, V_) if (pl.b == B_ && pl.v == V_) return mv_launch_n<MV_PLANES, B_, V_, false>(p, m, s);
    QNN_MV_CASE(1, 1) QNN_MV_CASE(1, 2) QNN_MV_CASE(1, 4)
    QNN_MV_CASE(2, 1) QNN_MV_CASE(2, 2) QNN_MV_CASE(2, 4)
    QNN_MV_CASE(3, 1) QNN_MV_CASE(3, 2)
    QNN_MV_CASE(4, 1) QNN_MV_CASE(4, 2)
#undef QNN_MV_CASE
    return QNN_ERR_UNSUPPORTED;
}

}  // namespace qnn
