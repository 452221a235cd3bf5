// Decoding of packed 4+4-bit samples into signed bytes, shared by the unpack
// kernels (unpack.cu) and the small-array X-engine (xeng_small.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace corr {
namespace {

__device__ __forceinline__ void decode_byte(uint32_t b, bool zero_invalid, int &r, int &m)
{
    r = ((int)(int8_t)(uint8_t)b) >> 4;             // high nibble, sign-extended
    m = ((int)(int8_t)(uint8_t)(b << 4)) >> 4;      // low nibble, sign-extended
    if (zero_invalid && (((b & 0xF0u) == 0x80u) || ((b & 0x0Fu) == 0x08u))) {
        r = 0;
        m = 0;
    }
}

__device__ __forceinline__ uint32_t pack4(int a, int b, int c, int d)
{
    return (uint32_t(a) & 0xFFu) | ((uint32_t(b) & 0xFFu) << 8) |
           ((uint32_t(c) & 0xFFu) << 16) | ((uint32_t(d) & 0xFFu) << 24);
}

// r, m and -m of the four packed samples of w, as four signed bytes each.  With
// u = nibble ^ 8 = value + 8 (0..15) in every byte, (u + 0x78) ^ 0x80 is the
// signed byte u - 8 and (0x88 - u) ^ 0x80 the signed byte 8 - u, and neither sum
// carries out of its byte.  A zero byte gives 0 + 0i.
__device__ __forceinline__ void decode4(uint32_t w, bool zero_invalid, uint32_t &R, uint32_t &M, uint32_t &N)
{
    const uint32_t ur = ((w >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
    const uint32_t um = (w & 0x0F0F0F0Fu) ^ 0x08080808u;
    R = (ur + 0x78787878u) ^ 0x80808080u;
    M = (um + 0x78787878u) ^ 0x80808080u;
    N = (0x88888888u - um) ^ 0x80808080u;
    if (zero_invalid) {
        // a nibble code of 8 (u == 0) in either part makes the sample 0 + 0i
        const uint32_t bad = __vcmpeq4(ur, 0u) | __vcmpeq4(um, 0u);
        R &= ~bad;
        M &= ~bad;
        N &= ~bad;
    }
}

// Byte k of X and byte k of Y for k = 0..3, interleaved as two words:
// lo = (X0, Y0, X1, Y1), hi = (X2, Y2, X3, Y3).
__device__ __forceinline__ void zip4(uint32_t X, uint32_t Y, uint32_t &lo, uint32_t &hi)
{
    lo = __byte_perm(X, Y, 0x5140);
    hi = __byte_perm(X, Y, 0x7362);
}

// From A = (a0, b0, a1, b1) and B = (c0, d0, c1, d1): (a0, b0, c0, d0) and (a1, b1, c1, d1).
__device__ __forceinline__ void pairs2(uint32_t A, uint32_t B, uint32_t &first, uint32_t &second)
{
    first = __byte_perm(A, B, 0x5410);
    second = __byte_perm(A, B, 0x7632);
}

// Four inputs' words (r(t), m(t), r(t+1), m(t+1)) and their twisted copies
// (-m(t), r(t), -m(t+1), r(t+1)) from the packed samples of the four inputs at
// t (w0) and t + 1 (w1).
__device__ __forceinline__ void words4(uint32_t w0, uint32_t w1, bool zero_invalid, uint32_t wa[4], uint32_t ww[4])
{
    uint32_t R0, M0, N0, R1, M1, N1;
    decode4(w0, zero_invalid, R0, M0, N0);
    decode4(w1, zero_invalid, R1, M1, N1);
    uint32_t a0, a1, b0, b1;
    zip4(R0, M0, a0, a1);
    zip4(R1, M1, b0, b1);
    pairs2(a0, b0, wa[0], wa[1]);
    pairs2(a1, b1, wa[2], wa[3]);
    zip4(N0, R0, a0, a1);
    zip4(N1, R1, b0, b1);
    pairs2(a0, b0, ww[0], ww[1]);
    pairs2(a1, b1, ww[2], ww[3]);
}

}  // namespace
}  // namespace corr
