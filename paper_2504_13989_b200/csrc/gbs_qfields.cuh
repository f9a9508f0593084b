// Packed codes -> int8 operands of the quantized matmul's integer contractions.
#pragma once

namespace {

// 32 two's-complement fields of a row (BITS words) become eight words of four int8, in pairs.  No sign extension is computed: a field
// moved to the TOP bits of its byte is the int8 value q * 2^(8 - BITS) (the field's sign bit becomes the byte's), products are then
// scaled by a power of two that the epilogue's scale factor takes out exactly, and the int32 sums stay far below 2^31 (49 * d' * 2^10
// at most).  A dot product does not see the order of its terms, only that both operands use the same one:
//   * Four bits on both sides: pair o is the even and the odd fields of word o (a mask; a shift and a mask).
//   * Three bits on a side: an octet of fields is three bytes, so the bytes are gathered first, one octet per byte lane (six byte
//     permutes).  Field e of all four octets then moves to the top of its lane in one shift and one mask, or two of each where it
//     straddles two bytes: 25 operations for 32 fields, where spreading every octet to nibbles took 56.  Four-bit codes opposite are
//     transposed likewise (eight permutes).
// 4096 x 4096 x 4096 with 3 bits on both sides: 89 us when every octet was spread, 75 now; 16 tokens: 9.5 -> 6.5.
template <int BITS>
__device__ __forceinline__ void gather_octets(const unsigned w[BITS], unsigned p[BITS])
{
    if (BITS == 3) {
        p[0] = __byte_perm(__byte_perm(w[0], w[1], 0x0630), w[2], 0x5210);      // bytes 0, 3, 6, 9
        p[1] = __byte_perm(__byte_perm(w[0], w[1], 0x0741), w[2], 0x6210);      //       1, 4, 7, 10
        p[2] = __byte_perm(__byte_perm(w[0], w[1], 0x0052), w[2], 0x7410);      //       2, 5, 8, 11
    } else {
        const unsigned a = __byte_perm(w[0], w[1], 0x5140), b = __byte_perm(w[2], w[BITS - 1], 0x5140);
        const unsigned c = __byte_perm(w[0], w[1], 0x7362), d = __byte_perm(w[2], w[BITS - 1], 0x7362);
        p[0] = __byte_perm(a, b, 0x5410);
        p[1] = __byte_perm(a, b, 0x7632);
        p[2] = __byte_perm(c, d, 0x5410);
        p[BITS - 1] = __byte_perm(c, d, 0x7632);
    }
}
// pair o, o < 4, of gathered words (fields 2 o and 2 o + 1 of the four octets) or of four-bit words as they are
template <int BITS>
__device__ __forceinline__ void field_pair(const unsigned p[BITS], int o, unsigned& even, unsigned& odd)
{
    if (BITS == 4) {
        even = (p[o < BITS ? o : 0] << 4) & 0xf0f0f0f0u;
        odd = p[o < BITS ? o : 0] & 0xf0f0f0f0u;
    } else if (o == 0) {
        even = (p[0] << 5) & 0xe0e0e0e0u;
        odd = (p[0] << 2) & 0xe0e0e0e0u;
    } else if (o == 1) {
        even = ((p[0] >> 1) & 0x60606060u) | ((p[1] << 7) & 0x80808080u);
        odd = (p[1] << 4) & 0xe0e0e0e0u;
    } else if (o == 2) {
        even = (p[1] << 1) & 0xe0e0e0e0u;
        odd = ((p[1] >> 2) & 0x20202020u) | ((p[2] << 6) & 0xc0c0c0c0u);
    } else {
        even = (p[2] << 3) & 0xe0e0e0e0u;
        odd = p[2] & 0xe0e0e0e0u;
    }
}

}  // namespace
