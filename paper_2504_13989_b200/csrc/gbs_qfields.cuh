// Packed codes -> int8 operands of the quantized matmul's integer contractions.
#pragma once

namespace {

// Eight two's-complement fields (24 or 32 bits) -> two words of four int8 each: the even fields, the odd fields.
// No sign extension is computed: a field moved to the TOP bits of its byte is the int8 value q * 2^(8 - BITS) (the
// field's sign bit becomes the byte's), products are then scaled by a power of two that the epilogue's scale factor
// takes out exactly, and the int32 sums stay far below 2^31 (49 * d' * 2^10 at most).  Four-bit fields already sit in
// nibbles: one mask for the odd ones, a shift and a mask for the even ones.  Three-bit fields are first spread to one
// per nibble by three mask-and-shift steps.
template <int BITS>
__device__ __forceinline__ void fields_to_int8(unsigned f, unsigned& even, unsigned& odd)
{
    if (BITS == 4) {
        odd = f & 0xf0f0f0f0u;
        even = (f << 4) & 0xf0f0f0f0u;
    } else {
        f = (f & 0x00000fffu) | ((f & 0x00fff000u) << 4);       // 12 bits per half-word
        f = (f & 0x003f003fu) | ((f & 0x0fc00fc0u) << 2);       // 6 bits per byte
        f = (f & 0x07070707u) | ((f & 0x38383838u) << 1);       // 3 bits per nibble (bit 3 of every nibble clear)
        odd = (f << 1) & 0xe0e0e0e0u;
        even = (f << 5) & 0xe0e0e0e0u;
    }
}

}  // namespace
