// C ABI entry points: host-side validation, size queries and dispatch.
// Every step of the path itself runs in the kernels of the sibling files.
#include <stdlib.h>

#include "common.cuh"

namespace qnn {

std::atomic<unsigned long long> g_launches{0};

int sm_count() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
            n = 148;
        cached[dev] = n;
    }
    return cached[dev];
}

static bool valid_fmt(int fmt) { return fmt == QNN_FMT_BITPLANES || fmt == QNN_FMT_INT8; }
static int field_bits(int bits) { return bits == 1 ? 1 : (bits == 2 ? 2 : 4); }

static qnn_status check_gemm_desc(const qnn_gemm_desc *d, bool has_thr, int *path_out) {
    if (!d) return QNN_ERR_INVALID_ARG;
    if (d->M <= 0 || d->N <= 0 || d->K <= 0) return QNN_ERR_INVALID_ARG;
    if (d->w_bits < 1 || d->w_bits > 8 || d->a_bits < 1 || d->a_bits > 8) return QNN_ERR_INVALID_ARG;
    if (!(valid_fmt(d->w_fmt) || d->w_fmt == QNN_FMT_FIELDS) || !valid_fmt(d->a_fmt)) return QNN_ERR_INVALID_ARG;
    if (d->w_enc < 0 || d->w_enc > 2 || d->a_enc < 0 || d->a_enc > 2) return QNN_ERR_INVALID_ARG;
    if (d->path < QNN_PATH_AUTO || d->path > QNN_PATH_TCGEN05_I8) return QNN_ERR_INVALID_ARG;
    if (d->skip_planes < 0) return QNN_ERR_INVALID_ARG;
    // leaving plane pairs out is a notion of the bit-plane formulation only
    if (d->skip_planes > 0 && (d->w_fmt != QNN_FMT_BITPLANES || d->a_fmt != QNN_FMT_BITPLANES)) return QNN_ERR_UNSUPPORTED;
    if (has_thr) {
        if (d->out_bits < 1 || d->out_bits > 4) return QNN_ERR_INVALID_ARG;
        if (!valid_fmt(d->out_fmt)) return QNN_ERR_INVALID_ARG;
    }
    if (!valid_enc(d->w_enc, d->w_bits) || !valid_enc(d->a_enc, d->a_bits)) return QNN_ERR_UNSUPPORTED;
    if (d->w_fmt == QNN_FMT_FIELDS) {
        // packed w-bit weights against 8-bit activation containers: the few-column kernel only
        if (d->a_fmt != QNN_FMT_INT8 || d->path == QNN_PATH_BITSERIAL) return QNN_ERR_UNSUPPORTED;
        if (!gemv_fields_dp4a_fits(d) && !gemv_fields_fits(d, has_thr)) return QNN_ERR_UNSUPPORTED;
        if (path_out) *path_out = QNN_PATH_TCGEN05_I8;
        return QNN_OK;
    }
    if (d->w_fmt != d->a_fmt) return QNN_ERR_UNSUPPORTED;
    int path = d->path;
    if (path == QNN_PATH_AUTO)
        path = d->w_fmt == QNN_FMT_INT8 ? QNN_PATH_TCGEN05_I8 : QNN_PATH_BITSERIAL;
    if (path == QNN_PATH_TCGEN05_I8 && d->w_fmt != QNN_FMT_INT8) return QNN_ERR_UNSUPPORTED;
    if (path == QNN_PATH_BITSERIAL) {
        if (d->w_fmt != QNN_FMT_BITPLANES) return QNN_ERR_UNSUPPORTED;
        if (d->w_bits > 4 || d->a_bits > 4) return QNN_ERR_UNSUPPORTED;
    }
    // int32 accumulator range: K * max|w| * max|a| must stay below 2^31
    const double wmax = d->w_enc == QNN_ENC_BIPOLAR ? 1.0
                        : (d->w_enc == QNN_ENC_SIGNED ? double(1 << (d->w_bits - 1)) : double((1 << d->w_bits) - 1));
    const double amax = d->a_enc == QNN_ENC_BIPOLAR ? 1.0
                        : (d->a_enc == QNN_ENC_SIGNED ? double(1 << (d->a_bits - 1)) : double((1 << d->a_bits) - 1));
    if (double(d->K) * wmax * amax >= 2147483648.0) return QNN_ERR_UNSUPPORTED;
    if (path_out) *path_out = path;
    return QNN_OK;
}

static qnn_status check_conv_desc(const qnn_conv_desc *d) {
    if (!d) return QNN_ERR_INVALID_ARG;
    if (d->B <= 0 || d->H <= 0 || d->W <= 0 || d->C <= 0 || d->OC <= 0 || d->KH <= 0 || d->KW <= 0)
        return QNN_ERR_INVALID_ARG;
    if (d->stride <= 0 || d->pad < 0 || d->in_pitch < 0) return QNN_ERR_INVALID_ARG;
    if (!valid_fmt(d->fmt)) return QNN_ERR_INVALID_ARG;
    if (d->a_bits < 1 || d->a_bits > 8) return QNN_ERR_INVALID_ARG;
    if (d->H + 2 * d->pad < d->KH || d->W + 2 * d->pad < d->KW) return QNN_ERR_INVALID_ARG;
    // the lowered GEMM's column count B*OH*OW and the map's pixel count are ints
    const long long oh = (d->H + 2 * d->pad - d->KH) / d->stride + 1, ow = (d->W + 2 * d->pad - d->KW) / d->stride + 1;
    if ((long long)d->B * oh * ow > 0x7fffffffll || (long long)d->B * d->H * d->W > 0x7fffffffll)
        return QNN_ERR_UNSUPPORTED;
    if (d->fmt == QNN_FMT_INT8 && d->in_pitch != 0 && d->in_pitch < d->C) return QNN_ERR_INVALID_ARG;
    if (d->a_enc == QNN_ENC_BIPOLAR && d->pad > 0) return QNN_ERR_UNSUPPORTED;
    // per-pixel pad bits would read as -1 for a bipolar operand
    if (d->fmt == QNN_FMT_BITPLANES && (d->C % 32) != 0 &&
        (d->a_enc == QNN_ENC_BIPOLAR || d->w_enc == QNN_ENC_BIPOLAR) &&
        (d->a_enc == QNN_ENC_BIPOLAR) == (d->w_enc == QNN_ENC_BIPOLAR))
        return QNN_ERR_UNSUPPORTED;
    return QNN_OK;
}

static void conv_to_gemm(const qnn_conv_desc *d, qnn_gemm_desc *g) {
    g->M = d->OC;
    g->N = d->B * qnn_conv_out_h(d) * qnn_conv_out_w(d);
    g->K = qnn_conv_lowered_k(d);
    g->w_bits = d->w_bits; g->a_bits = d->a_bits; g->out_bits = d->out_bits;
    g->w_enc = d->w_enc; g->a_enc = d->a_enc;
    g->w_fmt = d->fmt; g->a_fmt = d->fmt; g->out_fmt = d->out_fmt;
    g->path = d->path;
    g->skip_planes = 0;
}

// Bit planes with more columns than the few-column kernel takes go through the tensor cores, expanded
// to bytes inside the kernel, unless the caller asks for the bit-serial path or leaves plane pairs
// out.  Sixteen plane pairs (W4A4) up to 2^30 multiply-accumulates keep the AND/POPC kernel although
// dense operands take longer there (1024^3: 156 us against 20): that a call gets faster with
// skip_planes and with empty plane tiles is what this format promises at these sizes.
static bool planes_on_tensor_cores(const qnn_gemm_desc *d) {
    if (d->path != QNN_PATH_AUTO || d->skip_planes != 0) return false;
    // The roles of a tensor-core CTA wait for each other at most 2e9 cycles, and the epilogue waits for a
    // whole tile: 3500 cycles per 128 elements of the depth (four planes each), 0.9e9 at 2^25.  AND/POPC
    // waits for nothing.
    if (d->K > (1 << 25)) return false;
    const double macs = (double)d->M * d->N * d->K;
    // a single plane pair at middle sizes (512^3: 7.6 us against 10.9; 1024^3: 16.0 against 13.5)
    if (d->w_bits * d->a_bits == 1 && macs > double(1 << 24) && macs <= double(1 << 27)) return false;
    return d->w_bits * d->a_bits < 16 || macs > double(1 << 30);
}

// Whether the tensor-core kernel that expands planes inside beats the AND/POPC kernel, which it does not
// where few plane pairs meet little work, raw sums or many thresholds: an estimate of both in microseconds.
// AND/POPC: 64 x 64 tiles, two CTAs per SM, 512 elements of the depth a step; tensor cores: 128 x 128 tiles
// whose depth two CTAs share when there are few, 128 elements a step, an epilogue that grows with the
// thresholds and with raw rows that are not whole 16-byte units, and in a convolution word-by-word copies
// unless pixels are whole 16-byte units.  Fitted to 3800 random products and 2900 convolutions of one to
// four plane pairs, replayed as a graph; call after call the AND/POPC kernel, which is launched normally,
// takes 1.9 us more (the launch gap), the other 0.5, and 1.8 us are added so that neither kind of caller
// loses.  On 5762 others the choice costs 0.7 % (graph) and 0.3 % (calls) of the faster one's time on average, always the
// tensor cores 2.6 % and 1.2 % (325 x 313 x 132 W1A1 raw sums: 14.5 us there, 6.2 with AND/POPC), always
// AND/POPC 105 %.  From five plane pairs on the tensor cores were the faster ones everywhere.
static bool planes_tensor_faster(const qnn_gemm_desc *d, const qnn_conv_desc *cv, bool has_thr) {
    const int planes = d->w_bits + d->a_bits, pairs = d->w_bits * d->a_bits, sms = sm_count();
    if (pairs > 4) return true;
    const double ctas = (double)ceil_div(d->M, 64) * ceil_div(d->N, 64), waves = (double)(((long long)ctas + 2 * sms - 1) / (2 * sms));
    const int steps = ceil_div(ceil_div(d->K, 32), 16);
    const double counted = 2.9 + 1.8 + waves * steps * (2.7 * pairs + 0.14 * planes) + ctas * (8.5e-3 + 5.1e-3 * steps * pairs) +
                           (has_thr ? 1.65 : 0.0) + (has_thr && d->out_fmt == QNN_FMT_BITPLANES ? 0.84 * d->out_bits : 0.0);
    const long long tiles = (long long)ceil_div(d->M, 128) * ceil_div(d->N, 128);
    const int kb = ceil_div(d->K, 128);
    const bool share = 2 * tiles <= sms && kb >= 4, by_words = cv && ceil_div(cv->C, 32) % 4 != 0;
    const double rounds = share ? 1.0 : (double)((tiles + sms - 1) / sms);
    // epilogue of a tile by thresholds (1, 3, 7, 15) or raw sums, in the last round and in those before it
    static const double last_us[5] = {0.0, 1.5, 2.4, 4.9, 6.9}, more_us[5] = {0.0, 0.0, 0.0, 3.3, 3.3};
    const double last = has_thr ? last_us[d->out_bits] : (d->M % 4 ? 4.6 : 1.4), more = has_thr ? more_us[d->out_bits] : (d->M % 4 ? 8.3 : 2.5);
    const double part = d->M < 128 ? ceil_div(d->M, 32) / 4.0 : 1.0;
    const double tensor = 4.3 + (cv ? 0.9 : 0.0) + (by_words ? 3.3 : 0.0) + (share ? 2.7 : 0.0) + part * last + (rounds - 1.0) * (3.5 + part * more) +
                          rounds * (share ? ceil_div(kb, 2) : kb) * (0.47 + (by_words ? 0.2 : 0.11) * planes);
    return counted > 0.95 * tensor;
}

// The kernel a valid problem runs on: the one place where qnn_qgemm and the host queries decide.
enum Route {
    ROUTE_FIELDS_MMA, ROUTE_FIELDS_DP4A, ROUTE_FIELDS_TENSOR,      // packed weights
    ROUTE_BYTES_MMA, ROUTE_BYTES_DP4A, ROUTE_TENSOR,               // 8-bit containers
    ROUTE_PLANES_MMA, ROUTE_PLANES_POPC, ROUTE_PLANES_TENSOR, ROUTE_PLANES_TILED
};
static Route gemm_route(const qnn_gemm_desc *d, bool has_thr, int path) {
    if (d->w_fmt == QNN_FMT_FIELDS) {
        if (!getenv("QNN_FIELDS_KERNEL") && gemv_mma_takes(d, has_thr)) return ROUTE_FIELDS_MMA;
        // one column: byte dot products on the CUDA cores, where it fits their shared memory; else the tcgen05 form
        return gemv_fields_dp4a_fits(d) ? ROUTE_FIELDS_DP4A : ROUTE_FIELDS_TENSOR;
    }
    // 8-bit containers with a handful of columns and no path forced: the weights are streamed once
    // (a tensor-core tile would be almost empty)
    if (d->path == QNN_PATH_AUTO && d->w_fmt == QNN_FMT_INT8 && gemv_i8_fits(d))
        return gemv_mma_takes(d, has_thr) ? ROUTE_BYTES_MMA : ROUTE_BYTES_DP4A;
    if (path == QNN_PATH_TCGEN05_I8) return ROUTE_TENSOR;
    // a handful of columns: stream the weight planes once ...
    if (gemv_planes_fits(d))
        // ... on the tensor cores, unless the caller asks for the bit-serial path or leaves pairs out
        return d->path == QNN_PATH_AUTO && d->skip_planes == 0 && gemv_mma_takes(d, has_thr) ? ROUTE_PLANES_MMA : ROUTE_PLANES_POPC;
    return planes_on_tensor_cores(d) && planes_tensor_faster(d, nullptr, has_thr) ? ROUTE_PLANES_TENSOR : ROUTE_PLANES_TILED;
}

// Convolution on bit planes by way of 8-bit containers: the map and the filters are widened into the
// workspace, which has room for them wherever a lowered matrix would be several times the map, and the
// 8-bit convolution kernels run on that.  Expanding inside the GEMM kernel instead repeats the work
// for every filter tap of the map and every pixel tile of the filters, and pays only where the extra
// launch weighs more (27 x 27 x 96 -> 256, 5 x 5, W1A2 at batch 8: 15 us this way, 38 in the kernel).
constexpr double WIDEN_MIN_MACS = double(1 << 28);
static qnn_status widened_conv_launch(const qnn_conv_desc *d, const qnn_gemm_desc *g, const void *Wp, const void *in,
                                      const int32_t *thr, void *out, void *ws, size_t ws_bytes, cudaStream_t s) {
    const int Cp = round_up(d->C, 16);
    const long long pixels = (long long)d->B * d->H * d->W, taps = (long long)d->OC * d->KH * d->KW;
    if (pixels * Cp > 0x7fffffffffffll || taps > 0x7fffffffll || pixels > 0x7fffffffll) return QNN_ERR_UNSUPPORTED;
    const size_t map_bytes = ((size_t)pixels * Cp + 255) / 256 * 256, w_bytes = (size_t)taps * Cp;
    if (map_bytes + w_bytes > ws_bytes || (double)g->M * g->N * g->K < WIDEN_MIN_MACS) return QNN_ERR_UNSUPPORTED;
    qnn_conv_desc c = *d;
    c.C = Cp; c.in_pitch = Cp; c.fmt = QNN_FMT_INT8;
    qnn_gemm_desc cg = *g;
    cg.K = qnn_conv_lowered_k(&c); cg.w_fmt = cg.a_fmt = QNN_FMT_INT8;
    // a pixel's words widen to one row of Cp bytes, and so do a filter tap's
    const qnn_pack_desc pm = {(int)pixels, d->C, d->a_bits, d->a_enc, QNN_FMT_BITPLANES};
    const qnn_pack_desc pw = {(int)taps, d->C, d->w_bits, d->w_enc, QNN_FMT_BITPLANES};
    uint8_t *map = reinterpret_cast<uint8_t *>(ws), *filters = map + map_bytes;
    if (!gemm_tc_conv_takes(&c)) return QNN_ERR_UNSUPPORTED;
    qnn_status st = planes_to_int8_launch(&pm, in, map, s, &pw, Wp, filters);
    if (st == QNN_OK) st = gemm_tc_lower_launch(&c, &cg, filters, map, thr, out, s);
    if (st == QNN_ERR_UNSUPPORTED) st = gemm_tc_conv_launch(&c, &cg, filters, map, thr, out, true, s);
    return st;
}

}  // namespace qnn

using namespace qnn;

extern "C" {

int qnn_version(void) { return 100; }

const char *qnn_status_string(qnn_status s) {
    switch (s) {
        case QNN_OK: return "ok";
        case QNN_ERR_INVALID_ARG: return "invalid argument";
        case QNN_ERR_UNSUPPORTED: return "unsupported combination";
        case QNN_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
        case QNN_ERR_WORKSPACE: return "workspace missing or too small";
        case QNN_ERR_CUDA: return "CUDA call failed";
        case QNN_ERR_DEVICE_TIMEOUT: return "device-side wait timed out";
    }
    return "unknown status";
}

unsigned long long qnn_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

size_t qnn_packed_ld(int K, int fmt) {
    if (K <= 0) return 0;
    if (fmt == QNN_FMT_BITPLANES) return (size_t)ceil_div(K, 32);
    if (fmt == QNN_FMT_INT8) return (size_t)round_up(K, 16);
    return 0;           // QNN_FMT_FIELDS: the pitch depends on the bit width, see qnn_packed_bytes
}

size_t qnn_packed_bytes(const qnn_pack_desc *d) {
    if (!d || d->rows <= 0 || d->K <= 0 || d->bits < 1 || d->bits > 8) return 0;
    if (d->fmt == QNN_FMT_BITPLANES) return (size_t)d->bits * d->rows * qnn_packed_ld(d->K, d->fmt) * 4;
    if (d->fmt == QNN_FMT_INT8) return (size_t)d->rows * qnn_packed_ld(d->K, d->fmt);
    if (d->fmt == QNN_FMT_FIELDS && d->bits <= 4)
        return (size_t)d->rows * 32 * ceil_div(d->K, 32 * (8 / field_bits(d->bits)));
    return 0;
}

qnn_status qnn_pack(const qnn_pack_desc *d, const void *logical, void *packed, void *stream) {
    if (!d || !logical || !packed) return QNN_ERR_INVALID_ARG;
    if (d->rows <= 0 || d->K <= 0 || d->bits < 1 || d->bits > 8) return QNN_ERR_INVALID_ARG;
    if (!(valid_fmt(d->fmt) || d->fmt == QNN_FMT_FIELDS) || d->enc < 0 || d->enc > 2) return QNN_ERR_INVALID_ARG;
    if (!valid_enc(d->enc, d->bits)) return QNN_ERR_UNSUPPORTED;
    if (d->fmt == QNN_FMT_FIELDS && d->bits > 4) return QNN_ERR_UNSUPPORTED;
    if (!aligned16(logical) || !aligned16(packed)) return QNN_ERR_ALIGNMENT;
    return pack_launch(d, logical, packed, (cudaStream_t)stream);
}

qnn_status qnn_planes_to_int8(const qnn_pack_desc *d, const void *planes, void *containers, void *stream) {
    if (!d || !planes || !containers) return QNN_ERR_INVALID_ARG;
    if (d->rows <= 0 || d->K <= 0 || d->bits < 1 || d->bits > 8) return QNN_ERR_INVALID_ARG;
    if (d->fmt != QNN_FMT_BITPLANES || d->enc < 0 || d->enc > 2) return QNN_ERR_INVALID_ARG;
    if (!valid_enc(d->enc, d->bits)) return QNN_ERR_UNSUPPORTED;
    if (!aligned16(planes) || !aligned16(containers)) return QNN_ERR_ALIGNMENT;
    return planes_to_int8_launch(d, planes, containers, (cudaStream_t)stream);
}

size_t qnn_gemm_workspace_bytes(const qnn_gemm_desc *d) {
    int path = 0;
    if (check_gemm_desc(d, true, &path) != QNN_OK) return 0;
    if (d->w_fmt != QNN_FMT_INT8 || path != QNN_PATH_TCGEN05_I8) return 0;
    if (d->path == QNN_PATH_AUTO && gemv_i8_fits(d)) return 0;
    return gemm_tc_workspace_bytes(d);
}

size_t qnn_gemm_out_bytes(const qnn_gemm_desc *d, int has_thresholds) {
    if (!d || d->M <= 0 || d->N <= 0) return 0;
    if (!has_thresholds) return (size_t)d->N * d->M * 4;
    if (d->out_fmt == QNN_FMT_INT8) return (size_t)d->N * round_up(d->M, 16);
    if (d->out_fmt == QNN_FMT_BITPLANES) return (size_t)d->out_bits * d->N * ceil_div(d->M, 32) * 4;
    return 0;
}

int qnn_qgemm_kernel(const qnn_gemm_desc *d, int has_thresholds) {
    int path = 0;
    const qnn_status st = check_gemm_desc(d, has_thresholds != 0, &path);
    if (st != QNN_OK) return (int)st;
    switch (gemm_route(d, has_thresholds != 0, path)) {
        case ROUTE_FIELDS_MMA: case ROUTE_FIELDS_DP4A: case ROUTE_FIELDS_TENSOR: return QNN_KERNEL_FIELDS_FEW_COLUMNS;
        case ROUTE_BYTES_MMA: case ROUTE_BYTES_DP4A: return QNN_KERNEL_BYTES_FEW_COLUMNS;
        case ROUTE_TENSOR: return gemm_tc_uses_pair_kernel(d) ? QNN_KERNEL_TENSOR_CTA_PAIR : QNN_KERNEL_TENSOR;
        case ROUTE_PLANES_MMA: case ROUTE_PLANES_POPC: return QNN_KERNEL_PLANES_FEW_COLUMNS;
        case ROUTE_PLANES_TENSOR: case ROUTE_PLANES_TILED: break;
    }
    return QNN_KERNEL_PLANES_TILED;
}

const char *qnn_qgemm_kernel_name(const qnn_gemm_desc *d, int has_thresholds) {
    int path = 0;
    if (check_gemm_desc(d, has_thresholds != 0, &path) != QNN_OK) return nullptr;
    switch (gemm_route(d, has_thresholds != 0, path)) {
        case ROUTE_FIELDS_MMA: case ROUTE_BYTES_MMA: case ROUTE_PLANES_MMA: return "gemv_mma_kernel";
        case ROUTE_FIELDS_DP4A: return "gemv_fields_dp4a_kernel";
        case ROUTE_FIELDS_TENSOR: return "gemv_fields_kernel";
        case ROUTE_BYTES_DP4A: return "gemv_i8_kernel";
        case ROUTE_TENSOR: return gemm_tc_uses_pair_kernel(d) ? "qgemm_tc2_kernel" : "qgemm_tc_kernel";
        case ROUTE_PLANES_POPC: return "gemv_planes_kernel";
        case ROUTE_PLANES_TENSOR: return "qgemm_tc_kernel";
        case ROUTE_PLANES_TILED: break;
    }
    return "qgemm_bitserial_kernel";
}

qnn_status qnn_qgemm(const qnn_gemm_desc *d, const void *W, const void *A, const int32_t *thr,
                     void *out, void *workspace, size_t workspace_bytes, void *stream) {
    int path = 0;
    qnn_status st = check_gemm_desc(d, thr != nullptr, &path);
    if (st != QNN_OK) return st;
    if (!W || !A || !out) return QNN_ERR_INVALID_ARG;
    if (!aligned16(W) || !aligned16(A) || !aligned16(out) || !aligned4(thr))
        return QNN_ERR_ALIGNMENT;
    const cudaStream_t cs = (cudaStream_t)stream;
    switch (gemm_route(d, thr != nullptr, path)) {
        case ROUTE_FIELDS_MMA: case ROUTE_BYTES_MMA: case ROUTE_PLANES_MMA: return gemv_mma_launch(d, W, A, thr, out, cs);
        case ROUTE_FIELDS_DP4A: return gemv_fields_dp4a_launch(d, W, A, thr, out, cs);
        case ROUTE_FIELDS_TENSOR: return gemv_fields_launch(d, W, A, thr, out, cs);
        case ROUTE_BYTES_DP4A: return gemv_i8_launch(d, W, A, thr, out, cs);
        case ROUTE_TENSOR: {
            // the workspace is optional (see the header): used only when given, large enough and aligned
            const bool ws_ok = workspace && aligned16(workspace);
            return gemm_tc_launch(d, W, A, thr, out, ws_ok ? workspace : nullptr, ws_ok ? workspace_bytes : 0, cs);
        }
        case ROUTE_PLANES_POPC: return gemv_planes_launch(d, W, A, thr, out, cs);
        case ROUTE_PLANES_TENSOR:
            st = gemm_tc_planes_launch(nullptr, d, W, A, thr, out, cs);
            if (st != QNN_ERR_UNSUPPORTED) return st;
            break;
        case ROUTE_PLANES_TILED: break;
    }
    return gemm_bitserial_launch(d, W, A, thr, out, cs);
}

int qnn_conv_out_h(const qnn_conv_desc *d) {
    return d ? (d->H + 2 * d->pad - d->KH) / d->stride + 1 : 0;
}
int qnn_conv_out_w(const qnn_conv_desc *d) {
    return d ? (d->W + 2 * d->pad - d->KW) / d->stride + 1 : 0;
}

int qnn_conv_lowered_k(const qnn_conv_desc *d) {
    if (!d) return 0;
    if (d->fmt == QNN_FMT_BITPLANES) return 32 * d->KH * d->KW * ceil_div(d->C, 32);
    if (d->C % 16 == 0) return d->KH * d->KW * d->C;
    return d->KH * round_up(d->KW * d->C, 16);       // one zero-padded run per filter row
}

size_t qnn_conv_lowered_bytes(const qnn_conv_desc *d) {
    if (check_conv_desc(d) != QNN_OK) return 0;
    qnn_pack_desc p;
    p.rows = d->B * qnn_conv_out_h(d) * qnn_conv_out_w(d);
    p.K = qnn_conv_lowered_k(d);
    p.bits = d->a_bits; p.enc = d->a_enc; p.fmt = d->fmt;
    return qnn_packed_bytes(&p);
}

size_t qnn_conv_workspace_bytes(const qnn_conv_desc *d) {
    size_t b = qnn_conv_lowered_bytes(d);
    return (b + 255) / 256 * 256;
}

size_t qnn_conv_out_bytes(const qnn_conv_desc *d, int has_thresholds) {
    if (check_conv_desc(d) != QNN_OK) return 0;
    qnn_gemm_desc g;
    conv_to_gemm(d, &g);
    return qnn_gemm_out_bytes(&g, has_thresholds);
}

qnn_status qnn_im2col(const qnn_conv_desc *d, const void *in, void *lowered, void *stream) {
    qnn_status st = check_conv_desc(d);
    if (st != QNN_OK) return st;
    if (!in || !lowered) return QNN_ERR_INVALID_ARG;
    if (!aligned16(in) || !aligned16(lowered)) return QNN_ERR_ALIGNMENT;
    return im2col_launch(d, in, lowered, (cudaStream_t)stream);
}

qnn_status qnn_qconv(const qnn_conv_desc *d, const void *Wpacked, const void *in, const int32_t *thr,
                     void *out, void *workspace, size_t workspace_bytes, void *stream) {
    qnn_status st = check_conv_desc(d);
    if (st != QNN_OK) return st;
    qnn_gemm_desc g;
    conv_to_gemm(d, &g);
    int path = 0;
    st = check_gemm_desc(&g, thr != nullptr, &path);
    if (st != QNN_OK) return st;
    if (!Wpacked || !in || !out) return QNN_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < qnn_conv_workspace_bytes(d)) return QNN_ERR_WORKSPACE;
    if (!aligned16(Wpacked) || !aligned16(in) || !aligned16(out) || !aligned16(workspace) || !aligned4(thr))
        return QNN_ERR_ALIGNMENT;
    // 8-bit maps on the tensor-core path: the GEMM's loader does the lowering itself (im2col
    // tensor map) where the shape allows; QNN_CONV_EXPLICIT=1 in the environment keeps the
    // lowered matrix (measurements, tests)
    const char *explicit_env = getenv("QNN_CONV_EXPLICIT");
    if (path == QNN_PATH_TCGEN05_I8 && !(explicit_env && explicit_env[0] == '1')) {
        // three-channel maps whose rows shared memory holds: nothing is lowered
        st = conv_direct_launch(d, &g, Wpacked, in, thr, out, false, (cudaStream_t)stream);
        if (st != QNN_ERR_UNSUPPORTED) return st;
        // lowering warps inside the kernel where the tensor-map loader does not apply (few
        // channels: other first layers) or would waste k-blocks (channel count not a multiple of 128)
        st = gemm_tc_lower_launch(d, &g, Wpacked, in, thr, out, (cudaStream_t)stream);
        if (st != QNN_ERR_UNSUPPORTED) return st;
        st = gemm_tc_conv_launch(d, &g, Wpacked, in, thr, out, false, (cudaStream_t)stream);
        if (st != QNN_ERR_UNSUPPORTED) return st;
    }
    // bit-plane maps on the tiled bit-serial kernel: its staging code lowers on the fly (a handful
    // of output pixels goes through the lowered matrix and the few-column kernel instead)
    if (path == QNN_PATH_BITSERIAL && !(explicit_env && explicit_env[0] == '1') && !gemv_planes_fits(&g)) {
        if (planes_on_tensor_cores(&g)) {
            st = widened_conv_launch(d, &g, Wpacked, in, thr, out, workspace, workspace_bytes, (cudaStream_t)stream);
            if (st != QNN_ERR_UNSUPPORTED) return st;
            if (planes_tensor_faster(&g, d, thr != nullptr)) {
                st = gemm_tc_planes_launch(d, &g, Wpacked, in, thr, out, (cudaStream_t)stream);
                if (st != QNN_ERR_UNSUPPORTED) return st;
            }
        }
        st = gemm_bitserial_conv_launch(d, &g, Wpacked, in, thr, out, (cudaStream_t)stream);
        if (st != QNN_ERR_UNSUPPORTED) return st;
    }
    st = im2col_launch(d, in, workspace, (cudaStream_t)stream);
    if (st != QNN_OK) return st;
    return qnn_qgemm(&g, Wpacked, workspace, thr, out, nullptr, 0, stream);
}

int qnn_conv_boxes(const qnn_conv_desc *d, int has_thresholds, int *w, int *h, int *n) {
    qnn_gemm_desc g;
    int path = 0;
    if (check_conv_desc(d) != QNN_OK || !w || !h || !n) return 0;
    conv_to_gemm(d, &g);
    if (check_gemm_desc(&g, has_thresholds != 0, &path) != QNN_OK || path != QNN_PATH_TCGEN05_I8) return 0;
    return gemm_tc_conv_boxes(d, &g, has_thresholds != 0, w, h, n);
}

int qnn_conv_in_place(const qnn_conv_desc *d, int has_thresholds) {
    qnn_gemm_desc g;
    int path = 0;
    if (check_conv_desc(d) != QNN_OK) return 0;
    conv_to_gemm(d, &g);
    if (check_gemm_desc(&g, has_thresholds != 0, &path) != QNN_OK || path != QNN_PATH_TCGEN05_I8) return 0;
    return conv_direct_takes(d, &g, has_thresholds != 0, false) ? 1 : 0;
}

int qnn_conv_maxpool_fuses(const qnn_conv_desc *d, int k, int stride) {
    qnn_gemm_desc g;
    int path = 0;
    if (check_conv_desc(d) != QNN_OK || k != 3 || stride != 2) return 0;
    conv_to_gemm(d, &g);
    if (check_gemm_desc(&g, true, &path) != QNN_OK || path != QNN_PATH_TCGEN05_I8) return 0;
    return conv_direct_takes(d, &g, true, true) ? 1 : 0;
}

qnn_status qnn_qconv_maxpool(const qnn_conv_desc *d, int k, int stride, const void *Wpacked, const void *in,
                             const int32_t *thr, void *out, void *stream) {
    qnn_status st = check_conv_desc(d);
    if (st != QNN_OK) return st;
    qnn_gemm_desc g;
    conv_to_gemm(d, &g);
    int path = 0;
    st = check_gemm_desc(&g, true, &path);
    if (st != QNN_OK) return st;
    if (!Wpacked || !in || !thr || !out || k <= 0 || stride <= 0) return QNN_ERR_INVALID_ARG;
    if (!aligned16(Wpacked) || !aligned16(in) || !aligned16(out) || !aligned4(thr)) return QNN_ERR_ALIGNMENT;
    if (k != 3 || stride != 2 || path != QNN_PATH_TCGEN05_I8) return QNN_ERR_UNSUPPORTED;
    return conv_direct_launch(d, &g, Wpacked, in, thr, out, true, (cudaStream_t)stream);
}

// Lowered-matrix storage of qnn_qconv_static.  In host code this name is only a
// handle for cudaGetSymbolAddress; the kernels get the address that call returns.
static __device__ __align__(256) unsigned char g_static_lowered[QNN_QCONV_STATIC_MAX_BYTES];

// Device address of g_static_lowered on the current device, looked up once per device.
static qnn_status static_lowered_ptr(void **ptr) {
    static void *cached[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return QNN_ERR_CUDA;
    if (!cached[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_lowered) != cudaSuccess || !p) return QNN_ERR_CUDA;
        cached[dev] = p;
    }
    *ptr = cached[dev];
    return QNN_OK;
}

qnn_status qnn_qconv_static(const qnn_conv_desc *d, const void *Wpacked, const void *in, const int32_t *thr,
                            void *out, void *stream) {
    qnn_status st = check_conv_desc(d);
    if (st != QNN_OK) return st;
    qnn_gemm_desc g;
    conv_to_gemm(d, &g);
    st = check_gemm_desc(&g, thr != nullptr, nullptr);
    if (st != QNN_OK) return st;
    if (qnn_conv_workspace_bytes(d) > (size_t)QNN_QCONV_STATIC_MAX_BYTES) return QNN_ERR_WORKSPACE;
    if (!Wpacked || !in || !out) return QNN_ERR_INVALID_ARG;
    if (!aligned16(Wpacked) || !aligned16(in) || !aligned16(out) || !aligned4(thr)) return QNN_ERR_ALIGNMENT;
    void *lowered = nullptr;
    st = static_lowered_ptr(&lowered);
    if (st != QNN_OK) return st;
    st = im2col_launch(d, in, lowered, (cudaStream_t)stream);
    if (st != QNN_OK) return st;
    return qnn_qgemm(&g, Wpacked, lowered, thr, out, nullptr, 0, stream);
}

qnn_status qnn_maxpool(const qnn_pool_desc *d, const void *in, void *out, void *stream) {
    if (!d || !in || !out) return QNN_ERR_INVALID_ARG;
    if (d->B <= 0 || d->H <= 0 || d->W <= 0 || d->C <= 0 || d->k <= 0 || d->stride <= 0)
        return QNN_ERR_INVALID_ARG;
    if (d->k > d->H || d->k > d->W) return QNN_ERR_INVALID_ARG;
    if (d->bits < 1 || d->bits > 8 || !valid_fmt(d->fmt)) return QNN_ERR_INVALID_ARG;
    if (d->fmt == QNN_FMT_BITPLANES && d->bits > 4) return QNN_ERR_UNSUPPORTED;
    if (!aligned16(in) || !aligned16(out)) return QNN_ERR_ALIGNMENT;
    return maxpool_launch(d, in, out, (cudaStream_t)stream);
}

qnn_status qnn_validate_thresholds(const int32_t *thr, int M, int n_thr, int *n_bad_rows, void *stream) {
    if (!thr || !n_bad_rows || M <= 0 || n_thr <= 0) return QNN_ERR_INVALID_ARG;
    return validate_thresholds_launch(thr, M, n_thr, n_bad_rows, (cudaStream_t)stream);
}

qnn_status qnn_device_status(int *status) {
    if (!status) return QNN_ERR_INVALID_ARG;
    return device_status_read(status);
}

}  // extern "C"
