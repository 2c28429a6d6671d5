// Bit planes (Section 3.1) widened to bytes in registers, for the kernels that multiply them on the
// tensor cores.
//
// A 32-element word of every plane of a row becomes eight registers: bit j + 8 i of a word is byte i of
// register j, so each register is one shift and one AND away from a word of 1-, 2- or 4-bit fields.
// Both operands go through the same permutation of the depth, which leaves the product alone.
#pragma once

#include "common.cuh"

namespace qnn {

enum { PL_UNSIGNED = 0, PL_SIGNED = 1, PL_BIPOLAR = 2 };

// Words of a row of B planes -> 32 bytes (eight registers).  Planes are first merged into 2-bit,
// then 4-bit fields (3.5 instructions per register for four planes instead of 8).  A signed value
// is offset binary once its top plane is flipped; 2^(B-1) comes off each byte with the byte's top
// bit set as a borrow guard.  +-1: 1 - 2 * (bit clear), one multiply-add.
template <int B, int KIND>
__device__ __forceinline__ void expand_word(const uint32_t *w, uint32_t (&o)[8]) {
    if (KIND == PL_BIPOLAR) {
#pragma unroll
        for (int j = 0; j < 8; ++j) o[j] = ((~w[0] >> j) & 0x01010101u) * 0xFEu + 0x01010101u;
        return;
    }
    constexpr uint32_t TOP = KIND == PL_SIGNED ? 0xFFFFFFFFu : 0u;
    constexpr uint32_t GUARD = KIND == PL_SIGNED ? 0x80808080u : 0u;
    if (B == 1) {
        const uint32_t x = w[0] ^ TOP;
#pragma unroll
        for (int j = 0; j < 8; ++j) o[j] = ((x >> j) & 0x01010101u) | GUARD;
    } else {
        const uint32_t w1 = B == 2 ? w[1] ^ TOP : w[1];
        // 2-bit fields: even elements in e[0], odd ones in e[1]
        const uint32_t e[2] = {(w[0] & 0x55555555u) | ((w1 << 1) & 0xAAAAAAAAu), ((w[0] >> 1) & 0x55555555u) | (w1 & 0xAAAAAAAAu)};
        if (B == 2) {
#pragma unroll
            for (int j = 0; j < 8; ++j) o[j] = ((e[j & 1] >> (j & ~1)) & 0x03030303u) | GUARD;
        } else {
            const uint32_t w2 = B == 3 ? w[2] ^ TOP : w[2], w3 = B == 4 ? w[3] ^ TOP : 0u;
            const uint32_t f[2] = {(w2 & 0x55555555u) | ((w3 << 1) & 0xAAAAAAAAu), ((w2 >> 1) & 0x55555555u) | (w3 & 0xAAAAAAAAu)};
            // 4-bit fields: x[q] holds elements q, q + 4, q + 8, ...
            const uint32_t x[4] = {(e[0] & 0x33333333u) | ((f[0] << 2) & 0xCCCCCCCCu), (e[1] & 0x33333333u) | ((f[1] << 2) & 0xCCCCCCCCu),
                                   ((e[0] >> 2) & 0x33333333u) | (f[0] & 0xCCCCCCCCu), ((e[1] >> 2) & 0x33333333u) | (f[1] & 0xCCCCCCCCu)};
#pragma unroll
            for (int j = 0; j < 8; ++j) o[j] = ((x[j & 3] >> (j & 4)) & 0x0F0F0F0Fu) | GUARD;
        }
    }
    if (KIND == PL_SIGNED) {
#pragma unroll
        for (int j = 0; j < 8; ++j) o[j] = (o[j] - 0x01010101u * (1u << (B - 1))) ^ 0x80808080u;
    }
}

inline int plane_kind(int enc) {
    return enc == QNN_ENC_BIPOLAR ? PL_BIPOLAR : (enc == QNN_ENC_SIGNED ? PL_SIGNED : PL_UNSIGNED);
}

}  // namespace qnn
