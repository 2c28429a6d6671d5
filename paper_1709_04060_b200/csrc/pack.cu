// Operand packer: logical bytes -> bit planes (Section 3.1: plane i = bit i of
// every element, packed along the depth) or zero-padded 8-bit containers
// (Section 3: operands cast to 8-bit integers); bit planes -> 8-bit containers (few-bit data
// crosses the host link packed and is widened on the device).  Also the threshold validator.
#include "common.cuh"

namespace qnn {

// Bits i, 8+i, 16+i, 24+i of x gathered into the low nibble.
__device__ __forceinline__ uint32_t gather_bit4(uint32_t x, int i) {
    return (((x >> i) & 0x01010101u) * 0x01020408u) >> 24;
}

// One thread per (row, depth word): reads up to 32 logical bytes, writes one
// word into each plane.
template <bool BIPOLAR>
__global__ void pack_planes_kernel(const uint8_t *__restrict__ logical, uint32_t *__restrict__ planes,
                                   int rows, int K, int kw, int bits, bool vec_ok) {
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)rows * kw) return;
    const int r = (int)(idx / kw);
    const int w = (int)(idx - (long long)r * kw);
    const int k0 = w * 32;
    const uint8_t *src = logical + (size_t)r * K + k0;
    uint32_t x[8];
    if (vec_ok && k0 + 32 <= K) {
        const uint4 lo = *reinterpret_cast<const uint4 *>(src);
        const uint4 hi = *reinterpret_cast<const uint4 *>(src + 16);
        x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w;
        x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uint32_t v = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int k = k0 + q * 4 + b;
                if (k < K) v |= (uint32_t)src[q * 4 + b] << (8 * b);
            }
            x[q] = v;
        }
    }
    if (BIPOLAR) {
        // bit = (value > 0) per signed byte; zero pad bytes give bit 0
        uint32_t word = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t pos = __vcmpgts4(x[q], 0u) & 0x01010101u;
            word |= gather_bit4(pos, 0) << (4 * q);
        }
        planes[(size_t)r * kw + w] = word;
    } else {
        for (int i = 0; i < bits; ++i) {
            uint32_t word = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) word |= gather_bit4(x[q], i) << (4 * q);
            planes[((size_t)i * rows + r) * kw + w] = word;
        }
    }
}

// Per-byte conversion of four logical bytes to their 8-bit containers.
__device__ __forceinline__ uint32_t container4(uint32_t x, int bits, int enc) {
    if (enc == QNN_ENC_BIPOLAR) {
        const uint32_t gt = __vcmpgts4(x, 0u);                  // 0xFF where the byte is > 0
        return (gt & 0x01010101u) | ~gt;                        // +1 : -1
    }
    if (bits == 8) return x;
    const uint32_t low = x & (0x01010101u * ((1u << bits) - 1u));
    if (enc == QNN_ENC_UNSIGNED) return low;
    // sign extension inside every byte: the sign bit, moved up one place, times
    // 2^(8-bits) - 1 fills bits [bits, 8) and cannot carry into the next byte
    const uint32_t sign = low & (0x01010101u << (bits - 1));
    return low | ((sign << 1) * ((1u << (8 - bits)) - 1u));
}

// Bit planes -> 8-bit containers: one thread per plane word, i.e. 32 consecutive depth indices and two
// 16-byte stores (one where the row ends in the word's first half).  Four bits of a plane become four
// bytes by one multiplication (bit b of the nibble lands in bit 0 of byte b); plane i adds them shifted
// by i.  Bound by the stores at large sizes (16384 x 8192, four planes: 38 us = 5.3 TB/s) and by one
// load's latency and the fetch of the code at small ones.  A lone operand has a kernel for each number of
// planes, whose loads leave together, in CTAs of 128 threads (against one loop over the planes and 256
// threads: 378 x 494, six planes 2.5 -> 1.8 us; 4096 x 4096, four planes 6.9 -> 5.9).  The map and the
// filters of a convolution share a launch, which keeps the loop and the larger CTAs: the tensor-core
// kernel behind it is placed while this one drains, and twice the CTAs (13 x 16 x 10 x 128 -> 149, 3 x 3,
// W1A4, call after call: 10.5 -> 11.2 us) or more code (11.4) delay that.
struct WidenOp {
    const uint32_t *planes;
    uint4 *packed;
    long long words;           // rows * kw
    int K, kw, chunks, bits, enc;
};
template <int BITS>       // p.bits, or 0: a loop over them
__device__ __forceinline__ void widen_word(const WidenOp &p, long long idx) {
    long long r;
    if (p.words <= 0x7fffffffll) r = (unsigned)idx / (unsigned)p.kw; else r = idx / p.kw;
    const int c = (int)(idx - r * p.kw), k0 = 32 * c;
    uint32_t o[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) o[q] = 0u;
    auto load = [&](int i) { return __ldg(p.planes + i * p.words + idx); };
    auto add = [&](int i, uint32_t x) {
        // SIGNED: the top plane is the sign, which also fills the container's upper bits
        const uint32_t mul = (p.enc == QNN_ENC_SIGNED && i == p.bits - 1) ? ((0xFFu << i) & 0xFFu) : (1u << i);
#pragma unroll
        for (int q = 0; q < 8; ++q) o[q] |= ((((x >> (4 * q)) & 0xFu) * 0x00204081u) & 0x01010101u) * mul;
    };
    if (BITS > 0) {
        uint32_t w[BITS > 0 ? BITS : 1];
#pragma unroll
        for (int i = 0; i < BITS; ++i) w[i] = load(i);
#pragma unroll
        for (int i = 0; i < BITS; ++i) add(i, w[i]);
    } else {
#pragma unroll 4
        for (int i = 0; i < p.bits; ++i) add(i, load(i));
    }
    if (p.enc == QNN_ENC_BIPOLAR) {
        // bit 1 -> +1, bit 0 -> -1; pad bytes past K stay zero
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            uint32_t v = 0xFFFFFFFFu ^ (o[q] * 0xFEu);
            const int left = p.K - (k0 + 4 * q);                   // elements of this register inside the row
            if (left < 4) v &= left <= 0 ? 0u : (0xFFFFFFFFu >> (8 * (4 - left)));
            o[q] = v;
        }
    }
    uint4 *dst = p.packed + r * p.chunks + 2 * c;
    dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
    if (2 * c + 1 < p.chunks) dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
}
constexpr int WIDEN_THREADS = 128, WIDEN_PAIR_THREADS = 256;
template <int BITS>
__global__ void __launch_bounds__(WIDEN_THREADS) planes_to_int8_kernel(const WidenOp a) {
    pdl_trigger();        // a tensor-core kernel queued behind may set up while this one drains
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.words; i += step) widen_word<BITS>(a, i);
}
__global__ void __launch_bounds__(WIDEN_PAIR_THREADS) planes_to_int8_pair_kernel(const WidenOp a, const WidenOp b) {
    pdl_trigger();
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < a.words + b.words; i += step) {
        if (i < a.words) widen_word<0>(a, i); else widen_word<0>(b, i - a.words);
    }
}

// K a multiple of 16 (no padding): one thread per 16 bytes, 16-byte loads and stores.
__global__ void __launch_bounds__(256) pack_int8_vec_kernel(const uint4 *__restrict__ logical,
                                                            uint4 *__restrict__ packed, long long n16,
                                                            int bits, int enc) {
    pdl_trigger();        // a tensor-core kernel queued behind the packer may set up while it drains
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n16;
         i += (long long)gridDim.x * blockDim.x) {
        const uint4 v = logical[i];
        packed[i] = make_uint4(container4(v.x, bits, enc), container4(v.y, bits, enc),
                               container4(v.z, bits, enc), container4(v.w, bits, enc));
    }
}

// One thread per 16 output bytes of the [rows][ld] container matrix.
__global__ void pack_int8_kernel(const uint8_t *__restrict__ logical, uint8_t *__restrict__ packed,
                                 int rows, int K, int ld, int bits, int enc) {
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int chunks = ld / 16;
    if (idx >= (long long)rows * chunks) return;
    const int r = (int)(idx / chunks);
    const int c = (int)(idx - (long long)r * chunks);
    const uint8_t *src = logical + (size_t)r * K + c * 16;
    uint32_t o[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t v = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int k = c * 16 + q * 4 + b;
            uint32_t e = 0;
            if (k < K) {
                const uint32_t raw = src[q * 4 + b];
                if (enc == QNN_ENC_BIPOLAR) {
                    e = ((int8_t)raw > 0) ? 0x01u : 0xFFu;
                } else if (enc == QNN_ENC_SIGNED) {
                    const int sh = 32 - bits;
                    e = (uint32_t)(((int32_t)(raw << sh)) >> sh) & 0xFFu;
                } else {
                    e = raw & ((1u << bits) - 1u);
                }
            }
            v |= e << (8 * b);
        }
        o[q] = v;
    }
    *reinterpret_cast<uint4 *>(packed + (size_t)r * ld + c * 16) = make_uint4(o[0], o[1], o[2], o[3]);
}

// QNN_FMT_FIELDS: one thread per packed 32-bit word.  Byte j of 32-byte group g of a row holds,
// at bit position f*s, the field of element 32*S*g + 32*s + j (S = 8/f fields per byte).
__global__ void pack_fields_kernel(const uint8_t *__restrict__ logical, uint32_t *__restrict__ packed,
                                   int rows, int K, int ldw, int bits, int enc, int f) {
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)rows * ldw) return;
    const int r = (int)(idx / ldw);
    const int w = (int)(idx - (long long)r * ldw);
    const int S = 8 / f;
    const int g = w >> 3, j0 = (w & 7) * 4;
    const uint8_t *src = logical + (size_t)r * K;
    uint32_t word = 0;
    for (int b = 0; b < 4; ++b)
        for (int s = 0; s < S; ++s) {
            const long long k = (long long)32 * S * g + 32 * s + j0 + b;
            if (k >= K) continue;
            const int raw = (int8_t)src[k];
            uint32_t u;
            if (enc == QNN_ENC_BIPOLAR) u = raw > 0 ? 1u : 0u;
            else if (enc == QNN_ENC_SIGNED) {
                const int sh = 32 - bits;
                u = (uint32_t)(((int32_t)((uint32_t)raw << sh) >> sh) + (1 << (bits - 1)));   // value - minimum
            } else u = (uint32_t)raw & ((1u << bits) - 1u);
            word |= u << (8 * b + f * s);
        }
    packed[idx] = word;
}

static WidenOp widen_op(const qnn_pack_desc *d, const void *planes, void *packed) {
    WidenOp p = {};
    if (!d) return p;
    p.planes = (const uint32_t *)planes; p.packed = (uint4 *)packed;
    p.K = d->K; p.kw = ceil_div(d->K, 32); p.chunks = round_up(d->K, 16) / 16;
    p.words = (long long)d->rows * p.kw;
    p.bits = d->enc == QNN_ENC_BIPOLAR ? 1 : d->bits; p.enc = d->enc;
    return p;
}
qnn_status planes_to_int8_launch(const qnn_pack_desc *d, const void *planes, void *packed, cudaStream_t s,
                                 const qnn_pack_desc *d2, const void *planes2, void *packed2) {
    const WidenOp a = widen_op(d, planes, packed), b = widen_op(d2, planes2, packed2);
    const int threads = d2 ? WIDEN_PAIR_THREADS : WIDEN_THREADS;
    const long long want = (a.words + b.words + threads - 1) / threads, cap = (long long)sm_count() * 16;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    if (d2) {
        planes_to_int8_pair_kernel<<<grid, threads, 0, s>>>(a, b);
    } else {
#define QNN_WIDEN_CASE(B_) case B_: planes_to_int8_kernel<B_><<<grid, threads, 0, s>>>(a); break;
        switch (a.bits) {
            QNN_WIDEN_CASE(1) QNN_WIDEN_CASE(2) QNN_WIDEN_CASE(3) QNN_WIDEN_CASE(4)
            QNN_WIDEN_CASE(5) QNN_WIDEN_CASE(6) QNN_WIDEN_CASE(7) QNN_WIDEN_CASE(8)
            default: return QNN_ERR_UNSUPPORTED;
        }
#undef QNN_WIDEN_CASE
    }
    count_launch();
    return launch_status();
}

qnn_status pack_launch(const qnn_pack_desc *d, const void *logical, void *packed, cudaStream_t s) {
    const int threads = 256;
    if (d->fmt == QNN_FMT_FIELDS) {
        const int f = d->bits == 1 ? 1 : (d->bits == 2 ? 2 : 4);
        const int ldw = 8 * ceil_div(d->K, 32 * (8 / f));           // words per packed row
        const long long total = (long long)d->rows * ldw;
        pack_fields_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, s>>>(
            (const uint8_t *)logical, (uint32_t *)packed, d->rows, d->K, ldw, d->bits, d->enc, f);
        count_launch();
        return launch_status();
    }
    if (d->fmt == QNN_FMT_BITPLANES) {
        const int kw = ceil_div(d->K, 32);
        const long long total = (long long)d->rows * kw;
        const unsigned blocks = (unsigned)((total + threads - 1) / threads);
        const bool vec_ok = (d->K % 16) == 0;
        if (d->enc == QNN_ENC_BIPOLAR)
            pack_planes_kernel<true><<<blocks, threads, 0, s>>>((const uint8_t *)logical, (uint32_t *)packed,
                                                               d->rows, d->K, kw, 1, vec_ok);
        else
            pack_planes_kernel<false><<<blocks, threads, 0, s>>>((const uint8_t *)logical, (uint32_t *)packed,
                                                                d->rows, d->K, kw, d->bits, vec_ok);
    } else {
        const int ld = round_up(d->K, 16);
        const long long total = (long long)d->rows * (ld / 16);
        if (d->K % 16 == 0) {
            const long long want = (total + threads - 1) / threads;
            const long long cap = (long long)sm_count() * 16;
            pack_int8_vec_kernel<<<(unsigned)(want < cap ? want : cap), threads, 0, s>>>(
                (const uint4 *)logical, (uint4 *)packed, total, d->bits, d->enc);
            count_launch();
            return launch_status();
        }
        const unsigned blocks = (unsigned)((total + threads - 1) / threads);
        pack_int8_kernel<<<blocks, threads, 0, s>>>((const uint8_t *)logical, (uint8_t *)packed,
                                                    d->rows, d->K, ld, d->bits, d->enc);
    }
    count_launch();
    return launch_status();
}

__global__ void validate_thresholds_kernel(const int32_t *__restrict__ thr, int M, int n_thr, int *n_bad) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    bool bad = false;
    for (int i = 1; i < n_thr; ++i) bad |= thr[(size_t)m * n_thr + i] < thr[(size_t)m * n_thr + i - 1];
    if (bad) atomicAdd(n_bad, 1);
}

// Counter for the validator; a file-scope device word so that no allocation is needed.
__device__ int g_bad_rows;

qnn_status validate_thresholds_launch(const int32_t *thr, int M, int n_thr, int *n_bad_host, cudaStream_t s) {
    int *dev_ptr = nullptr;
    if (cudaGetSymbolAddress((void **)&dev_ptr, g_bad_rows) != cudaSuccess) return QNN_ERR_CUDA;
    if (cudaMemsetAsync(dev_ptr, 0, sizeof(int), s) != cudaSuccess) return QNN_ERR_CUDA;
    validate_thresholds_kernel<<<ceil_div(M, 128), 128, 0, s>>>(thr, M, n_thr, dev_ptr);
    count_launch();
    if (cudaGetLastError() != cudaSuccess) return QNN_ERR_CUDA;
    if (cudaMemcpyAsync(n_bad_host, dev_ptr, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return QNN_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return QNN_ERR_CUDA;
    return QNN_OK;
}

}  // namespace qnn
