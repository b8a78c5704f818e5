// Four trits at a time: int8x4 words of a plane <-> 2-bit codes (trit + 1) in the low bits of the bytes.
#pragma once
#include "ptqtp_internal.h"

namespace ptqtp {

// Codes of four trits.  A byte outside {-1, 0, 1} is stored as trit 0 and sets `bad`.
__device__ __forceinline__ uint32_t codes_of(uint32_t v, bool& bad) {
    const uint32_t neg = (v >> 7) & 0x01010101u;
    const uint32_t x = v ^ (neg * 255u);                 // of valid bytes: 0 (-1 and 0) or 1
    if ((x & 0xfefefefeu) | (x & neg)) {
        bad = true;
        uint32_t q = 0u;
        for (int b = 0; b < 32; b += 8) {
            const uint32_t c = (uint32_t)((int)(int8_t)(v >> b) + 1);
            q |= (c > 2u ? 1u : c) << b;
        }
        return q;
    }
    return 0x01010101u + x - neg;                        // no borrow between bytes
}
// The code bytes of four columns of a row pair: fields (row, plane 1), (row, plane 2), (row + 1, plane 1), (row + 1, plane 2).
__device__ __forceinline__ uint32_t pair_word(uint32_t a, uint32_t b, uint32_t c, uint32_t d, bool& bad) {
    return codes_of(a, bad) | codes_of(b, bad) << 2 | codes_of(c, bad) << 4 | codes_of(d, bad) << 6;
}
__device__ __forceinline__ uint4 pair_words(const uint4& a, const uint4& b, const uint4& c, const uint4& d, bool& bad) {
    return make_uint4(pair_word(a.x, b.x, c.x, d.x, bad), pair_word(a.y, b.y, c.y, d.y, bad), pair_word(a.z, b.z, c.z, d.z, bad),
                      pair_word(a.w, b.w, c.w, d.w, bad));
}
// Field f of four code bytes as trits.
__device__ __forceinline__ uint32_t trits_of(uint32_t word, int f) {
    return ((((word >> (2 * f)) & 0x03030303u) | 0x80808080u) - 0x01010101u) ^ 0x80808080u;
}
__device__ __forceinline__ uint4 trits_of(const uint4& w, int f) {
    return make_uint4(trits_of(w.x, f), trits_of(w.y, f), trits_of(w.z, f), trits_of(w.w, f));
}

}  // namespace ptqtp
