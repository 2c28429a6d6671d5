// First-layer convolution (few channels, 8 bit) on the tensor cores without a lowered matrix, in memory or
// anywhere else: the rows of the image sit in shared memory so that the tensor core's operand descriptor
// does the lowering of Section 3.2.
//
// A tcgen05 operand without swizzle is made of 16-byte pieces: row r of the operand at
// (r / 8) * SBO + (r % 8) * 16, its two pieces of a 32-byte step LBO apart.  With SBO = 128 the rows lie at
// a 16-byte pitch, and if that is also the step between neighbouring output pixels, row r + 1 is the same
// window one output pixel further on: the windows overlap in memory and nothing is copied.  So a pixel of
// three channels is stored in 16 / stride bytes (4 at stride 4, the channels and a byte that meets zero
// weights), and the pieces of filter row kh are the ceil(KW / stride) units from the output pixel's on.
// Image rows that are `stride` apart belong to neighbouring output rows; they are kept in `stride` classes
// of rows at a pitch of 8 * group_units units, so that the next output row is again a multiple of SBO away
// and a tile of 128 operand rows covers whole output rows (55 of 64 operand rows carry a pixel in the
// 227 x 227 layer).  Pieces are paired into 32-byte steps within rows that share a slot, so that LBO is the
// same whatever the ring position: 33 pieces make 17 steps (11 x 11 x 3, stride 4).
//
// What bounds it: neither the tensor pipe (64 cycles per step of 128 rows, 1088 a tile) nor the issue slots of
// the threshold count (12 288 accumulators a tile, 6.75 instructions each on the FP32 pipe, some 1500 cycles)
// but the latency of the epilogue warps' own chain: a tile takes 3800 cycles.  227 x 227 -> 96, 11 x 11,
// stride 4, batch 256: 128 us in the kernel that builds every lowered row with four warps (4 600 warp
// instructions a tile against some 400 here), 97 here; with the pool behind it 151 us in two kernels, 101 here.
//
// Roles: warp 0 issues the MMAs (descriptors from a table in shared memory, eight at a time: one by one the
// table's latency takes 89 cycles an MMA); warp 1 asks for the image rows of later steps by bulk copies (they
// are contiguous); warps 2-5 turn them into ring slots; the next ones lay out the weights, then run the
// epilogue, one 32 x 32 part of a tile per warp; with the pool in the kernel, four more take the maxima
// from the codes of the last three tiles, which the epilogue leaves in shared memory.  Up to 832 threads leave 72 or 80 registers
// each: with two output bits 4 to 48 bytes are spilled, else none.
#include <math.h>

#include "tc_epilogue.cuh"
#include "tc_ptx.cuh"

namespace qnn {

constexpr int DC_RING = 4;              // ring of row steps
constexpr int DC_STAGE_WARPS = 4;
constexpr int DC_MAX_STEPS = 64;        // 32-byte steps of the depth
constexpr int DC_RAW = 4;               // steps of image rows in flight
constexpr int DC_STAGE0 = 2, DC_EPI0 = DC_STAGE0 + DC_STAGE_WARPS;      // first staging, epilogue warp
constexpr int DC_POOL_WARPS = 4, DC_CODES = 3;   // code tiles in shared memory
constexpr int DC_MAX_THREADS = 32 * (DC_EPI0 + 16 + DC_POOL_WARPS);
constexpr int DC_BATCH = 4;             // units of a row step per staging thread
constexpr int DC_W_BATCH = 5;           // pieces of weights per thread in flight

struct DcStep { uint32_t at; uint16_t lbo, slot; };        // first piece: offset in the slot's row, distance to the second, slot

struct DcParams {
    const uint8_t *in, *W;
    const int32_t *thr;
    void *out;
    int M, N, ld_out, count;               // as the other tcgen05 kernels (epilogue)
    int H, row_bytes;                      // image rows, bytes of one
    long long total;                       // bytes of the map
    int OH, OW, KH, KW, stride;
    int pieces;                            // 16-byte pieces of a filter row
    int row_units;                         // units of a staged row that carry data
    int groups;                            // operand groups (of eight rows) per output row
    int rows_tile;                         // output rows per tile
    int extra;                             // row steps a tile needs beyond its own
    int class_bytes, mirror;               // one class of the ring; slots repeated at its end
    int raw_bytes;                         // image rows of a step, as they are
    int tiles_image, tiles, per;           // tiles (POOL kernels: pooled rows) per image, in all, per CTA
    int w_ld, w_run; long long w_total;    // weight rows: pitch, bytes per filter row; size of the matrix
    int chunks;                            // 32-channel parts of the output
    int PH, PW;                            // pooled output
    int steps;
    uint32_t idesc;
    int *status;
    DcStep step[DC_MAX_STEPS];
};

struct DcSmem {
    uint64_t desc_a[DC_RING][DC_MAX_STEPS], desc_w[DC_MAX_STEPS];   // operand descriptors of the steps, by ring position
    uint64_t full[DC_RING], empty[DC_RING], tmem_full[2], tmem_empty[2];
    uint64_t w_full, codes_full[DC_CODES], codes_empty[DC_CODES], raw_full[DC_RAW], raw_empty[DC_RAW];
    uint32_t tmem_base;
    int abort_flag;
};

// Bytes of the ring, and what a tile's 128 operand rows read past its last slot (rows that carry no pixel).
__host__ __device__ inline int dc_row_bytes(const DcParams &p) { return (p.stride * p.class_bytes + 2048 + 16 * p.pieces + 127) & ~127; }

// Operand descriptor without swizzle: 8-row groups 128 bytes apart.
__device__ __forceinline__ uint64_t dc_desc(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}

// The four aligned words around the twelve bytes at `at`; nothing outside [0, total) is read.
__device__ __noinline__ uint4 dc_words_end(const uint8_t *base, long long a, long long total) {
    uint32_t x[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
    for (int i = 0; i < 16 && a + i < total; ++i) {
        const uint32_t v = (uint32_t)base[a + i] << (8 * (i & 3));
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] |= (i >> 2) == k ? v : 0u;
    }
    return make_uint4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void dc_words(const uint8_t *base, long long at, long long total, uint32_t (&x)[4]) {
    const long long a = at & ~3ll;
    if (a + 16 <= total) {
        const uint32_t *q = reinterpret_cast<const uint32_t *>(base + a);
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = ld_global(q + i);
    } else {
        const uint4 v = dc_words_end(base, a, total);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    }
}
// ... as four pixels of three channels, the fourth byte of each undefined.
__device__ __forceinline__ void dc_pixels(const uint32_t (&x)[4], int shift, uint32_t (&px)[4]) {
    const uint32_t y0 = __funnelshift_r(x[0], x[1], shift), y1 = __funnelshift_r(x[1], x[2], shift), y2 = __funnelshift_r(x[2], x[3], shift);
    px[0] = y0;
    px[1] = __funnelshift_r(y0, y1, 24);
    px[2] = __funnelshift_r(y1, y2, 16);
    px[3] = y2 >> 8;
}
// The 16 bytes of a unit: `stride` pixels of 16 / stride bytes each.  Bytes that hold no channel meet zero
// weights.
__device__ __forceinline__ uint4 dc_unit(const uint32_t (&px)[4], int stride) {
    if (stride == 4) return make_uint4(px[0], px[1], px[2], px[3]);
    if (stride == 2) return make_uint4(px[0], 0u, px[1], 0u);
    return make_uint4(px[0], 0u, 0u, 0u);
}

// The tiles of one CTA, image by image: f(image, first tile, end).  POOL: the CTA's pooled rows; row r takes
// tile r (two output rows) and the first row of tile r + 1.
template <bool POOL, typename F>
__device__ __forceinline__ void dc_segments(const DcParams &p, F f) {
    int i = blockIdx.x * p.per;
    const int end = min(i + p.per, p.tiles);
    while (i < end) {
        const int b = i / p.tiles_image, t = i - b * p.tiles_image, n = min(p.tiles_image - t, end - i);
        if (!f(b, t, t + n + (POOL ? 1 : 0))) return;
        i += n;
    }
}

template <int OUT_MODE, int OUT_BITS, bool POOL>
__global__ void __launch_bounds__(DC_MAX_THREADS - (POOL ? 0 : 32 * DC_POOL_WARPS), 1)
conv_direct_kernel(const __grid_constant__ DcParams p) {
    extern __shared__ uint8_t dc_smem[];
    constexpr int NT = thr_slots(OUT_BITS);
    constexpr bool UNARY = POOL && OUT_BITS <= 2;         // codes of up to two bits are pooled in unary
    uint8_t *const base = dc_smem + ((128u - (smem_u32(dc_smem) & 127u)) & 127u);
    const int channels = 32 * p.chunks, row_b = p.groups * 128, ring_slots = DC_RING * p.rows_tile;
    uint8_t *const rows_s = base;                                                   // [class][slot][unit]
    uint8_t *const w_s = rows_s + dc_row_bytes(p);                                  // [piece][channel]
    int *const thr_s = reinterpret_cast<int *>(w_s + (size_t)p.steps * 2 * channels * 16);
    DcSmem &sm = *reinterpret_cast<DcSmem *>(thr_s + channels * NT);
    uint8_t *const raw_s = reinterpret_cast<uint8_t *>(&sm) + ((sizeof(DcSmem) + 15) & ~size_t(15));
    uint8_t *const codes_s = raw_s + DC_RAW * p.raw_bytes;                          // POOL: codes of three tiles
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, epi_warps = 4 * p.chunks;
    volatile int *abort_flag = &sm.abort_flag;

    if (threadIdx.x == 0) {
        for (int s = 0; s < DC_RING; ++s) { mbar_init(&sm.full[s], DC_STAGE_WARPS); mbar_init(&sm.empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&sm.tmem_full[b], 1); mbar_init(&sm.tmem_empty[b], epi_warps); }
        for (int b = 0; b < DC_CODES; ++b) { mbar_init(&sm.codes_full[b], epi_warps); mbar_init(&sm.codes_empty[b], DC_POOL_WARPS); }
        for (int b = 0; b < DC_RAW; ++b) { mbar_init(&sm.raw_full[b], 1); mbar_init(&sm.raw_empty[b], DC_STAGE_WARPS); }
        mbar_init(&sm.w_full, epi_warps);
        sm.abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        tmem_alloc(&sm.tmem_base, 256);
        for (int i = lane; i < p.steps * DC_RING; i += 32) {
            const int r = i / p.steps, s = i - r * p.steps;
            int slot = r * p.rows_tile + p.step[s].slot;
            if (slot >= ring_slots) slot -= ring_slots;
            sm.desc_a[r][s] = dc_desc(smem_u32(rows_s) + p.step[s].at + (uint32_t)(slot * row_b), p.step[s].lbo);
            if (r == 0) sm.desc_w[s] = dc_desc(smem_u32(w_s) + (uint32_t)(s * 2 * channels * 16), (uint32_t)channels * 16u);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem_base = sm.tmem_base;

    if (warp == 0) {
        // ---------------------------------------------------------- MMA issuer
        if (lane == 0) {
            uint32_t tile = 0, n = 0;                     // tiles and row steps so far
            const bool ready = mbar_wait(&sm.w_full, 0, abort_flag, p.status);
            if (ready) dc_segments<POOL>(p, [&](int, int t0, int t1) -> bool {
                for (int t = t0; t < t1; ++t, ++tile, ++n) {
                    const uint32_t buf = tile & 1, last = n + p.extra;
                    if (!mbar_wait(&sm.tmem_empty[buf], ((tile >> 1) & 1) ^ 1, abort_flag, p.status)) return false;
                    if (!mbar_wait(&sm.full[last % DC_RING], (last / DC_RING) & 1, abort_flag, p.status)) return false;
                    tc_fence_after();
                    const uint32_t d = tmem_base + buf * 128;
                    const uint64_t *da = sm.desc_a[n % DC_RING], *dw = sm.desc_w;
#pragma unroll 1
                    for (int s0 = 0; s0 < p.steps; s0 += 8) {
                        uint64_t a[8], w[8];
#pragma unroll
                        for (int s = 0; s < 8; ++s) { a[s] = da[s0 + s]; w[s] = dw[s0 + s]; }     // (the tables hold whole eights)
#pragma unroll
                        for (int s = 0; s < 8; ++s)
                            if (s0 + s < p.steps) umma_i8(d, a[s], w[s], p.idesc, (s0 | s) != 0);
                    }
                    umma_commit(&sm.empty[n % DC_RING]);
                    umma_commit(&sm.tmem_full[buf]);
                }
                // the steps that the segment's last tile read beyond its own
                for (int e = 0; e < p.extra; ++e, ++n) umma_commit(&sm.empty[n % DC_RING]);
                return true;
            });
        }
        __syncwarp();
    } else if (warp == 1) {
        // --------------------------------------- image rows of the coming steps, as they are
        if (lane == 0) {
            const int step_rows = p.rows_tile * p.stride;
            uint32_t n = 0;
            bool ok = true;
            dc_segments<POOL>(p, [&](int b, int t0, int t1) -> bool {
                for (int i = 0; i < t1 - t0 + p.extra; ++i, ++n) {
                    const uint32_t r = n % DC_RAW;
                    if (!(ok = mbar_wait(&sm.raw_empty[r], ((n / DC_RAW) & 1) ^ 1, abort_flag, p.status))) return false;
                    const int ih0 = (t0 + i) * step_rows, rows = max(0, min(step_rows, p.H - ih0));
                    const long long at = ((long long)b * p.H + ih0) * p.row_bytes, from = at & ~15ll;
                    // whole 16-byte units inside the map; its last bytes by plain loads.  (A row's last unit runs
                    // into the next row, whose bytes meet zero weights.)
                    long long to = (at + (long long)rows * p.row_bytes + 15) & ~15ll;
                    uint8_t *dst = raw_s + r * p.raw_bytes;
                    if (to > p.total) {
                        to = p.total & ~15ll;
                        for (long long q = max(to, from); q < p.total; ++q) dst[q - from] = p.in[q];
                    }
                    const uint32_t bytes = rows > 0 && to > from ? (uint32_t)(to - from) : 0u;
                    mbar_arrive_expect_tx(&sm.raw_full[r], bytes);
                    if (bytes)
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                     ::"r"(smem_u32(dst)), "l"(p.in + from), "r"(bytes), "r"(smem_u32(&sm.raw_full[r])) : "memory");
                }
                return true;
            });
            // gave up: the copies in flight land before the CTA exits
            if (!ok)
                for (uint32_t k = n > DC_RAW ? n - DC_RAW : 0; k < n; ++k) mbar_wait(&sm.raw_full[k % DC_RAW], (k / DC_RAW) & 1, abort_flag, p.status);
        }
        __syncwarp();
    } else if (warp < DC_EPI0) {
        // ------------------------------------- image rows into the ring
        const int w = warp - DC_STAGE0, ublocks = (p.row_units + 31) >> 5, step_rows = p.rows_tile * p.stride;
        // this thread's units of a step: row (past the last one: none), offset in the map, place in the ring
        int row[DC_BATCH], rel[DC_BATCH], dst[DC_BATCH], slot[DC_BATCH];
#pragma unroll
        for (int k = 0; k < DC_BATCH; ++k) {
            const int item = w + k * DC_STAGE_WARPS, unit = (item % ublocks) * 32 + lane;
            row[k] = item / ublocks;
            slot[k] = row[k] / p.stride;
            rel[k] = row[k] * p.row_bytes + unit * p.stride * 3;
            dst[k] = (row[k] - slot[k] * p.stride) * p.class_bytes + slot[k] * row_b + unit * 16;
            if (row[k] >= step_rows || unit >= p.row_units) row[k] = 1 << 30;
        }
        uint32_t n = 0;
        dc_segments<POOL>(p, [&](int b, int t0, int t1) -> bool {
            for (int i = 0; i < t1 - t0 + p.extra; ++i, ++n) {
                const uint32_t r = n % DC_RING, rr = n % DC_RAW;
                const int ih0 = (t0 + i) * step_rows;
                const int odd = (int)((((long long)b * p.H + ih0) * p.row_bytes) & 15);
                if (!__all_sync(0xffffffffu, mbar_wait(&sm.raw_full[rr], (n / DC_RAW) & 1, abort_flag, p.status))) return false;
                uint4 u[DC_BATCH];
#pragma unroll
                for (int k = 0; k < DC_BATCH; ++k)
                    if (row[k] < p.H - ih0) {
                        const uint32_t *q = reinterpret_cast<const uint32_t *>(raw_s + rr * p.raw_bytes) + ((odd + rel[k]) >> 2);
                        uint32_t x[4], px[4];
#pragma unroll
                        for (int v = 0; v < 4; ++v) x[v] = q[v];
                        dc_pixels(x, ((odd + rel[k]) & 3) * 8, px);
                        u[k] = dc_unit(px, p.stride);
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.raw_empty[rr]);
                if (!__all_sync(0xffffffffu, mbar_wait(&sm.empty[r], ((n / DC_RING) & 1) ^ 1, abort_flag, p.status))) return false;
#pragma unroll
                for (int k = 0; k < DC_BATCH; ++k)
                    if (row[k] < p.H - ih0) {
                        uint8_t *q = rows_s + dst[k] + (int)r * p.rows_tile * row_b;
                        *reinterpret_cast<uint4 *>(q) = u[k];
                        // a tile that starts in the last slots runs on behind them
                        if (r == 0 && slot[k] < p.mirror) *reinterpret_cast<uint4 *>(q + ring_slots * row_b) = u[k];
                    }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // visible to the tensor core's reads
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.full[r]);
            }
            return true;
        });
    } else if (POOL && warp >= DC_EPI0 + epi_warps) {
        // ------------------- maxima: pooled row t - 1 is the whole of tile t - 1 and the first row of tile t
        if constexpr (POOL) {
            const int first_thread = 32 * (DC_EPI0 + epi_warps), pitch = channels + 16;      // + 16: eight lanes on different banks
            uint32_t tile = 0;
            dc_segments<POOL>(p, [&](int b, int t0, int t1) -> bool {
                for (int t = t0; t < t1; ++t, ++tile) {
                    const uint32_t cb = tile % DC_CODES, pb = (tile + DC_CODES - 1) % DC_CODES;
                    if (!__all_sync(0xffffffffu, mbar_wait(&sm.codes_full[cb], (tile / DC_CODES) & 1, abort_flag, p.status))) return false;
                    if (t > t0) {
                        const uint8_t *const here = codes_s + (int)cb * 128 * pitch, *const before = codes_s + (int)pb * 128 * pitch;
                        const long long first = ((long long)b * p.PH + t - 1) * p.PW;
                        auto most = [&](int pw, int at) -> uint4 {
                            const uint8_t *row0 = before + 2 * pw * pitch + at, *row2 = here + 2 * pw * pitch + at;
                            uint4 v[9], m = make_uint4(0, 0, 0, 0);
#pragma unroll
                            for (int k = 0; k < 9; ++k)
                                v[k] = *reinterpret_cast<const uint4 *>((k < 3 ? row0 : (k < 6 ? row0 + 8 * p.groups * pitch : row2)) + (k % 3) * pitch);
#pragma unroll
                            for (int k = 0; k < 9; ++k) {
                                m.x = UNARY ? m.x | v[k].x : __vmaxu4(m.x, v[k].x); m.y = UNARY ? m.y | v[k].y : __vmaxu4(m.y, v[k].y);
                                m.z = UNARY ? m.z | v[k].z : __vmaxu4(m.z, v[k].z); m.w = UNARY ? m.w | v[k].w : __vmaxu4(m.w, v[k].w);
                            }
                            if (UNARY && OUT_BITS == 2) {
                                auto code = [](uint32_t x) { return (x & 0x01010101u) + ((x >> 1) & 0x01010101u) + ((x >> 2) & 0x01010101u); };
                                m = make_uint4(code(m.x), code(m.y), code(m.z), code(m.w));
                            }
                            return m;
                        };
                        if (OUT_MODE == OUT_U8) {
                            const int units = p.ld_out >> 4;
                            for (int k = threadIdx.x - first_thread; k < p.PW * units; k += 32 * DC_POOL_WARPS) {
                                const int pw = k / units, u = k - pw * units;
                                reinterpret_cast<uint4 *>(reinterpret_cast<uint8_t *>(p.out) + (size_t)(first + pw) * p.ld_out)[u] = most(pw, 16 * u);
                            }
                        } else {
                            const long long plane = (long long)(p.N / (p.OH * p.OW)) * p.PH * p.PW * p.chunks;
                            for (int k = threadIdx.x - first_thread; k < p.PW * p.chunks; k += 32 * DC_POOL_WARPS) {
                                const int pw = k / p.chunks, c = k - pw * p.chunks;
                                const uint4 lo = most(pw, 32 * c), hi = most(pw, 32 * c + 16);
                                const uint32_t m[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                                for (int q = 0; q < OUT_BITS; ++q) {
                                    uint32_t bits = 0;
#pragma unroll
                                    for (int v = 0; v < 8; ++v) bits |= nibble_of_plane(m[v], q) << (4 * v);
                                    reinterpret_cast<uint32_t *>(p.out)[q * plane + (first + pw) * p.chunks + c] = bits;
                                }
                            }
                        }
                    }
                    // the tile before this one has been read for the last time (and, at the end, this one)
                    __syncwarp();
                    if (lane == 0) {
                        if (t > t0) mbar_arrive(&sm.codes_empty[pb]);
                        if (t == t1 - 1) mbar_arrive(&sm.codes_empty[cb]);
                    }
                }
                return true;
            });
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // first the thresholds and weights of this warp's 32 channels; the pieces, in the order of the steps, are
        // dealt to the four warps that share them
        const int chunk = (warp - DC_EPI0) >> 2, quad = warp & 3, r = quad * 32 + lane, c = chunk * 32 + lane;
        if (OUT_MODE != OUT_RAW && ((warp - DC_EPI0) & 3) == 0) stage_thresholds<OUT_BITS, (UNARY || OUT_BITS >= 3), true>(p, thr_s + chunk * 32 * NT, chunk * 32, 32, lane);
        for (int k0 = (warp - DC_EPI0) & 3; k0 < 2 * p.steps; k0 += 4 * DC_W_BATCH) {
            uint32_t x[DC_W_BATCH][4];
            int shift[DC_W_BATCH], kw0[DC_W_BATCH];
#pragma unroll
            for (int k = 0; k < DC_W_BATCH; ++k) {
                const int piece = k0 + 4 * k, s = min(piece >> 1, p.steps - 1);
                // which filter row and unit this piece is (the second of a step: LBO further on)
                const int off = (int)p.step[s].at + (piece & 1 ? (int)p.step[s].lbo : 0);
                const int cls = off / p.class_bytes, j = (off - cls * p.class_bytes) >> 4, kh = p.step[s].slot * p.stride + cls;
                kw0[k] = p.KW;                                     // nothing but zeros
                shift[k] = 0;
                x[k][0] = x[k][1] = x[k][2] = x[k][3] = 0u;
                if (piece < 2 * p.steps && c < p.M && kh < p.KH && j < p.pieces) {
                    const long long at = (long long)c * p.w_ld + kh * p.w_run + j * p.stride * 3;
                    dc_words(p.W, at, p.w_total, x[k]);
                    shift[k] = (int)(at & 3) * 8;
                    kw0[k] = j * p.stride;
                }
            }
#pragma unroll
            for (int k = 0; k < DC_W_BATCH; ++k) {
                const int piece = k0 + 4 * k;
                uint32_t px[4];
                dc_pixels(x[k], shift[k], px);
#pragma unroll
                for (int q = 0; q < 4; ++q) px[q] = kw0[k] + q < p.KW ? px[q] & 0x00FFFFFFu : 0u;
                if (piece < 2 * p.steps) *reinterpret_cast<uint4 *>(w_s + ((size_t)piece * channels + c) * 16) = dc_unit(px, p.stride);
            }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");               // visible to the tensor core's reads
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.w_full);
        if (OUT_MODE != OUT_RAW) asm volatile("bar.sync %0, 128;" ::"r"(1 + chunk) : "memory");
        const int i = r / (8 * p.groups), ow = r - i * 8 * p.groups;               // output row of the tile, pixel in it
        const bool px_ok = i < p.rows_tile && ow < p.OW;
        uint32_t tile = 0;
        dc_segments<POOL>(p, [&](int b, int t0, int t1) -> bool {
            for (int t = t0; t < t1; ++t, ++tile) {
                const uint32_t buf = tile & 1;
                if (!__all_sync(0xffffffffu, mbar_wait(&sm.tmem_full[buf], (tile >> 1) & 1, abort_flag, p.status))) return false;
                tc_fence_after();
                int acc[32];
                tmem_ld32_issue(tmem_base + buf * 128 + ((uint32_t)(quad * 32) << 16) + chunk * 32, acc);
                tmem_ld_wait(acc);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.tmem_empty[buf]);                   // the accumulators are in registers
                if constexpr (!POOL) {
                    const int oh = t * p.rows_tile + i;
                    epilogue_chunk<OUT_MODE, OUT_BITS, true>(p, thr_s + chunk * 32 * NT, acc, (b * p.OH + oh) * p.OW + ow, px_ok && oh < p.OH, chunk * 32);
                } else {
                    const uint32_t cb = tile % DC_CODES;
                    uint32_t packed[8];
                    count_chunk<OUT_BITS, UNARY, true>(p, thr_s + chunk * 32 * NT, acc, packed);
                    if (!__all_sync(0xffffffffu, mbar_wait(&sm.codes_empty[cb], ((tile / DC_CODES) & 1) ^ 1, abort_flag, p.status))) return false;
                    uint4 *o = reinterpret_cast<uint4 *>(codes_s + (int)cb * 128 * (channels + 16) + r * (channels + 16) + chunk * 32);
                    o[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                    o[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.codes_full[cb]);
                }
            }
            return true;
        });
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 256);
    }
}

// ------------------------------------------------------------------- host side
// Where this kernel is the faster one.  From five rounds of tiles (pooled rows) per SM on: setting up (weights laid
// out, first rows) takes 7 us of a launch.  227 x 227 -> 96, 11 x 11, us with the pool, the other kernels -> this
// one: batch 16 15.8 -> 15.0, 24 19.6 -> 20.4, 32 26.4 -> 22.4, 64 42.8 -> 33.9, 256 151 -> 101; batch 1 8.7 -> 10.3.
// And where enough of the 128 operand rows of a tile carry a pixel: the kernel with lowering warps packs its tiles
// densely and spends the same epilogue on each, but lowers every row (40 x 40 -> 8, 7 x 7, batch 78, half of the
// rows used: 9.3 there, 20.9 here; 19 x 91 -> 32, 11 x 11, stride 2, batch 398: 16.5 and 47).  The share that is
// enough depends on how long the epilogue takes (output bits, 32-channel parts).  The logarithm of the two times'
// ratio is fitted to 835 random layers and, with the pool, 1702, those near 1 weighing most; below 0.92 (with the
// pool 0.87) it is taken.  Raw sums are bound by their stores: 1.2 times as long here.
constexpr int DC_MIN_ROUNDS = 5;
static bool dc_faster(const DcParams &p, const qnn_conv_desc *cv, const qnn_gemm_desc *g, bool has_thr, bool pool) {
    if (p.tiles < (long long)DC_MIN_ROUNDS * sm_count()) return false;
    // +-1 weights against pad bytes: the kernel with lowering warps does not take them (0.5 of the time; with a pool
    // behind it the same, but up to 1.3 times as long where the epilogue counts 7 or 15 thresholds)
    if (g->w_enc == QNN_ENC_BIPOLAR && cv->KW * 3 % 16 != 0 && (!pool || g->out_bits <= 2)) return true;
    if (!has_thr) return false;
    static const double bits[2][4] = {{0.173, 0.112, 0.091, 0.0}, {0.038, 0.007, 0.038, 0.0}};
    static const double parts[2][4] = {{0.074, -0.049, -0.084, 0.0}, {0.095, -0.114, -0.079, 0.0}};
    static const double base[2] = {-0.292, -0.080}, tile[2] = {0.5, -0.547}, slope[2] = {0.477, 0.419};
    // row steps of a CTA: its tiles, and what the last one of an image reads beyond
    const double steps = p.per + ((double)p.per / p.tiles_image + 1.0) * (p.extra + (pool ? 1 : 0));
    const double used = (double)p.N / (128.0 * p.tiles) * p.per / steps;
    return base[pool] + bits[pool][g->out_bits - 1] + parts[pool][p.chunks - 1] + tile[pool] / p.per < slope[pool] * log(used);
}
// The layers this kernel takes: three channels in contiguous pixels, no padding, up to 128 output channels,
// a stride that divides 4, rows of up to 128 units.
static bool dc_plan(const qnn_conv_desc *cv, const qnn_gemm_desc *g, bool has_thr, bool pool, DcParams *p) {
    const int pitch = cv->in_pitch ? cv->in_pitch : round_up(cv->C, 16);
    if (cv->fmt != QNN_FMT_INT8 || cv->C != 3 || pitch != 3 || cv->pad != 0 || cv->OC > 128) return false;
    if (cv->stride != 1 && cv->stride != 2 && cv->stride != 4) return false;
    const int S = cv->stride, OH = qnn_conv_out_h(cv), OW = qnn_conv_out_w(cv);
    p->H = cv->H; p->OH = OH; p->OW = OW; p->KH = cv->KH; p->KW = cv->KW; p->stride = S;
    if ((long long)cv->B * OH * OW > 0x7fffffffll || (long long)cv->W * 3 * (64 + cv->KH) > 0x7fffffffll) return false;
    p->row_bytes = cv->W * 3;
    p->total = (long long)cv->B * cv->H * p->row_bytes;
    p->pieces = ceil_div(cv->KW, S);
    p->row_units = OW - 1 + p->pieces;
    if (p->row_units > 128 || p->pieces > 64) return false;
    p->groups = ceil_div(p->row_units, 8);
    // output rows per tile: what 128 operand rows hold, and what the staging threads fetch in one go
    const int ublocks = ceil_div(p->row_units, 32);
    p->rows_tile = 16 / p->groups;
    if (p->rows_tile > DC_STAGE_WARPS * DC_BATCH / (S * ublocks)) p->rows_tile = DC_STAGE_WARPS * DC_BATCH / (S * ublocks);
    if (p->rows_tile < 1) return false;
    const int slots = (cv->KH - 1) / S;                            // slots behind its own that an output row reads
    p->extra = ceil_div(slots, p->rows_tile);
    if (p->extra > DC_RING - 2) return false;
    p->mirror = p->rows_tile - 1;
    // (units at the end of the last row read up to 12 bytes each behind it)
    p->raw_bytes = round_up(p->rows_tile * S * p->row_bytes + 16 + 12 * p->pieces + 16, 128);
    p->class_bytes = (DC_RING * p->rows_tile + p->mirror) * p->groups * 128;
    if (p->class_bytes > 0xffff) return false;
    p->chunks = ceil_div(cv->OC, 32);
    // 32-byte steps: the same piece of two filter rows that share a slot, else neighbouring pieces of one
    p->steps = 0;
    auto add = [&](int kh, int j, int lbo) {
        if (p->steps == DC_MAX_STEPS) return false;
        p->step[p->steps++] = {(uint32_t)((kh % S) * p->class_bytes + j * 16), (uint16_t)lbo, (uint16_t)(kh / S)};
        return true;
    };
    for (int kh = 0; kh < cv->KH; ++kh) {
        if (kh % S % 2 == 0 && kh % S + 1 < S && kh + 1 < cv->KH) {
            for (int j = 0; j < p->pieces; ++j)
                if (!add(kh, j, p->class_bytes)) return false;
            ++kh;
        } else {
            for (int j = 0; j < p->pieces; j += 2)
                if (!add(kh, j, 16)) return false;
        }
    }
    p->tiles_image = ceil_div(OH, p->rows_tile);
    if (pool) {
        if (p->rows_tile != 2 || OH < 3 || OW < 3) return false;
        p->PH = (OH - 3) / 2 + 1; p->PW = (OW - 3) / 2 + 1;
        p->tiles_image = p->PH;
    }
    const long long tiles = (long long)cv->B * p->tiles_image;
    if (tiles > 0x3fffffff) return false;
    p->tiles = (int)tiles;
    p->per = ceil_div(p->tiles, sm_count());
    p->M = g->M; p->N = g->N; p->ld_out = round_up(g->M, 16);
    if (!dc_faster(*p, cv, g, has_thr, pool)) return false;
    p->w_ld = round_up(g->K, 16); p->w_run = round_up(cv->KW * 3, 16);
    p->w_total = (long long)g->M * p->w_ld;
    const double wmax = g->w_enc == QNN_ENC_BIPOLAR ? 1.0
                        : (g->w_enc == QNN_ENC_SIGNED ? double(1 << (g->w_bits - 1)) : double((1 << g->w_bits) - 1));
    const double amax = g->a_enc == QNN_ENC_BIPOLAR ? 1.0
                        : (g->a_enc == QNN_ENC_SIGNED ? double(1 << (g->a_bits - 1)) : double((1 << g->a_bits) - 1));
    p->count = count_mode(double(cv->KH) * cv->KW * 3 * wmax * amax, true);
    p->idesc = (2u << 4) | ((g->a_enc == QNN_ENC_UNSIGNED ? 0u : 1u) << 7) | ((g->w_enc == QNN_ENC_UNSIGNED ? 0u : 1u) << 10) |
               ((uint32_t)(32 * p->chunks >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    return true;
}

static size_t dc_smem_bytes(const DcParams &p, int out_bits, bool pool) {
    const int channels = 32 * p.chunks;
    return 128 + (size_t)dc_row_bytes(p) + (size_t)p.steps * 2 * channels * 16 + (size_t)channels * thr_slots(out_bits) * 4 +
           sizeof(DcSmem) + 16 + (size_t)DC_RAW * p.raw_bytes + (pool ? (size_t)DC_CODES * 128 * (channels + 16) : 0);
}

template <int OUT_MODE, int OUT_BITS, bool POOL>
static qnn_status dc_launch(const DcParams &p, size_t smem, cudaStream_t s) {
    auto kern = conv_direct_kernel<OUT_MODE, OUT_BITS, POOL>;
    static std::atomic<bool> attr_done[QNN_MAX_DEVICES];           // per instantiation and device
    const int dev = current_device();
    if (dev < 0 || !allow_smem(kern, SMEM_LIMIT, attr_done[dev])) return QNN_ERR_CUDA;
    // programmatic dependent launch: at most one CTA more than the kernel ahead left room for is placed on an
    // SM early, and nothing is read before griddepcontrol.wait
    const int threads = 32 * (DC_EPI0 + 4 * p.chunks + (POOL ? DC_POOL_WARPS : 0));
    if (launch_pdl<DcParams>(kern, dim3((unsigned)ceil_div(p.tiles, p.per)), threads, smem, s, p) != cudaSuccess) return QNN_ERR_CUDA;
    count_launch();
    return launch_status();
}

bool conv_direct_takes(const qnn_conv_desc *cv, const qnn_gemm_desc *g, bool has_thr, bool pool) {
    DcParams p = {};
    return dc_plan(cv, g, has_thr, pool, &p) && (has_thr || !pool) && dc_smem_bytes(p, has_thr ? g->out_bits : 0, pool) <= SMEM_LIMIT;
}

// The convolution (UNSUPPORTED: the layer needs another kernel), with `pool` its 3 x 3, stride 2 max-pool too.
qnn_status conv_direct_launch(const qnn_conv_desc *cv, const qnn_gemm_desc *g, const void *W, const void *in,
                              const int32_t *thr, void *out, bool pool, cudaStream_t s) {
    DcParams p = {};
    if (!dc_plan(cv, g, thr != nullptr, pool, &p) || (pool && !thr)) return QNN_ERR_UNSUPPORTED;
    const size_t smem = dc_smem_bytes(p, thr ? g->out_bits : 0, pool);
    if (smem > SMEM_LIMIT) return QNN_ERR_UNSUPPORTED;
    p.in = (const uint8_t *)in; p.W = (const uint8_t *)W; p.thr = thr; p.out = out;
    p.status = device_status_word();
    if (!p.status) return QNN_ERR_CUDA;
    if (!thr) return dc_launch<OUT_RAW, 0, false>(p, smem, s);
#define QNN_DC_CASE(B_)                                                                                        \
    case B_:                                                                                                   \
        if (g->out_fmt == QNN_FMT_INT8) return pool ? dc_launch<OUT_U8, B_, true>(p, smem, s) : dc_launch<OUT_U8, B_, false>(p, smem, s); \
        return pool ? dc_launch<OUT_PLANES, B_, true>(p, smem, s) : dc_launch<OUT_PLANES, B_, false>(p, smem, s);
    switch (g->out_bits) { QNN_DC_CASE(1) QNN_DC_CASE(2) QNN_DC_CASE(3) QNN_DC_CASE(4) }
#undef QNN_DC_CASE
    return QNN_ERR_UNSUPPORTED;
}

}  // namespace qnn
