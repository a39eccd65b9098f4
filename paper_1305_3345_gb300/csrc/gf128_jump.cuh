// T * x^j in GF(2^128) (IEEE 1619's field, x^128 = x^7 + x^2 + x + 1, words
// little-endian) for a long jump, in a number of steps that grows with the
// length of j instead of j itself: x^j by squaring, then one multiplication.
// Squaring a polynomial over GF(2) spreads its bits to the even places.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace kgpu {
namespace dev {

// The low 16 bits of v, one to each even place.
__host__ __device__ __forceinline__ uint32_t spread_bits(uint32_t v) {
    v &= 0xFFFFu;
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    return (v | (v << 1)) & 0x55555555u;
}

// e <- e * x.
__host__ __device__ __forceinline__ void gf128_double(uint32_t (&e)[4]) {
    const uint32_t fold = (0u - (e[3] >> 31)) & 0x87u;
    e[3] = (e[3] << 1) | (e[2] >> 31);
    e[2] = (e[2] << 1) | (e[1] >> 31);
    e[1] = (e[1] << 1) | (e[0] >> 31);
    e[0] = (e[0] << 1) ^ fold;
}

// e <- e * e.
__host__ __device__ __forceinline__ void gf128_square(uint32_t (&e)[4]) {
    uint32_t h[4], l[4];
    for (int i = 0; i < 2; i++) {
        l[2 * i] = spread_bits(e[i]);
        l[2 * i + 1] = spread_bits(e[i] >> 16);
        h[2 * i] = spread_bits(e[i + 2]);
        h[2 * i + 1] = spread_bits(e[i + 2] >> 16);
    }
    // l + x^128 h = l + (x^7 + x^2 + x + 1) h, and what that shifts out again
    const uint32_t c = (h[3] >> 31) ^ (h[3] >> 30) ^ (h[3] >> 25);
    for (int i = 3; i > 0; i--)
        e[i] = l[i] ^ h[i] ^ (h[i] << 1 | h[i - 1] >> 31) ^ (h[i] << 2 | h[i - 1] >> 30) ^ (h[i] << 7 | h[i - 1] >> 25);
    e[0] = l[0] ^ h[0] ^ h[0] << 1 ^ h[0] << 2 ^ h[0] << 7 ^ c ^ c << 1 ^ c << 2 ^ c << 7;
}

// (w0, w1, w2, w3) <- that * x^j, j >= 64: at most 26 squarings, 13 at IEEE
// 1619's limit of 2^20 blocks a data unit, and the 128 steps of the
// multiplication.
__host__ __device__ __forceinline__ void gf128_jump(uint32_t& w0, uint32_t& w1, uint32_t& w2, uint32_t& w3,
                                                    uint32_t j) {
    uint32_t s = 0;
    while ((j >> s) > 127u) s++;
    const uint32_t top = j >> s;  // x^top is one bit
    uint32_t e[4];
    for (uint32_t i = 0; i < 4; i++) e[i] = top >> 5 == i ? 1u << (top & 31u) : 0u;
#pragma unroll 1
    while (s > 0) {
        gf128_square(e);
        if ((j >> --s) & 1u) gf128_double(e);
    }
    uint32_t r[4] = {0, 0, 0, 0};
#pragma unroll 1
    for (int i = 0; i < 128; i++) {  // Horner over the bits of e, highest first
        gf128_double(r);
        const uint32_t m = 0u - (e[3] >> 31);
        r[0] ^= w0 & m;
        r[1] ^= w1 & m;
        r[2] ^= w2 & m;
        r[3] ^= w3 & m;
        e[3] = (e[3] << 1) | (e[2] >> 31);
        e[2] = (e[2] << 1) | (e[1] >> 31);
        e[1] = (e[1] << 1) | (e[0] >> 31);
        e[0] <<= 1;
    }
    w0 = r[0];
    w1 = r[1];
    w2 = r[2];
    w3 = r[3];
}

}  // namespace dev
}  // namespace kgpu
