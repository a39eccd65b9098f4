// Bitsliced AES (FIPS-197) on 128 bit-planes of 32 blocks per thread: the
// pieces shared by the comparison variant (kgpu_bitslice.cu) and by the bulk
// kernels' bitsliced warps (kgpu_bulk.cu).  Plane 8p+b holds bit b of state
// byte p of all 32 blocks, one block per bit position; SubBytes is a Boolean
// circuit on 32-bit words (sbox_circuit.cuh), ShiftRows is a renaming of
// planes and MixColumns and AddRoundKey are XORs of planes.
#pragma once
#include <cstdint>

#include "sbox_circuit.cuh"

namespace kgpu {
namespace dev {

constexpr int kBsSpan = 1024;  // blocks per warp iteration (32 lanes x 32 blocks)

// In-place 32x32 bit transpose: afterwards bit t of a[k] is the former bit k of
// a[t].  Five rounds of block swaps (16, 8, 4, 2, 1); the 16- and 8-bit rounds
// are byte permutes.
__device__ __forceinline__ void transpose32(uint32_t* a) {
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t lo = a[i], hi = a[i + 16];
        a[i] = __byte_perm(lo, hi, 0x5410);
        a[i + 16] = __byte_perm(lo, hi, 0x7632);
    }
#pragma unroll
    for (int g = 0; g < 32; g += 16) {
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const uint32_t lo = a[g + i], hi = a[g + i + 8];
            a[g + i] = __byte_perm(lo, hi, 0x6240);
            a[g + i + 8] = __byte_perm(lo, hi, 0x7351);
        }
    }
#pragma unroll
    for (int s = 4; s >= 1; s >>= 1) {
        const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int i = 0; i < 32; i++) {
            if (i & s) continue;
            const uint32_t t = ((a[i] >> s) ^ a[i + s]) & m;
            a[i + s] ^= t;
            a[i] ^= t << s;
        }
    }
}

// One S-box circuit, called 16 times a round rather than inlined 16 times: the
// round body shrinks by ~1,500 instructions, which eases the instruction fetch
// stalls that top this kernel's profile (measured +4%, for 16 argument moves
// per call).
struct Byte8 {
    uint32_t x0, x1, x2, x3, x4, x5, x6, x7;
};

__device__ __noinline__ static Byte8 sbox_call(Byte8 b) {
    sbox_circuit(b.x0, b.x1, b.x2, b.x3, b.x4, b.x5, b.x6, b.x7);
    return b;
}

// The inverse of the S-box's affine map (FIPS-197 section 5.3.2): bit i of the
// result is x_(i+2) ^ x_(i+5) ^ x_(i+7), inverted for i = 0 and 2.
__device__ __forceinline__ void inverse_affine(uint32_t* x) {
    uint32_t y[8];
#pragma unroll
    for (int i = 0; i < 8; i++) y[i] = x[(i + 2) & 7] ^ x[(i + 5) & 7] ^ x[(i + 7) & 7];
    y[0] = ~y[0];
    y[2] = ~y[2];
#pragma unroll
    for (int i = 0; i < 8; i++) x[i] = y[i];
}

// InvSubBytes from the same circuit: with S = A o I, A the affine map and I
// the field inversion, which is its own inverse, S^-1 = I o A^-1 =
// A^-1 o S o A^-1.  Sixteen three-input XORs a byte more than SubBytes.
__device__ __forceinline__ void inv_sub_bytes(uint32_t (&S)[128]) {
#pragma unroll
    for (int p = 0; p < 16; p++) {
        uint32_t* x = S + 8 * p;
        inverse_affine(x);
        sbox_circuit(x[0], x[1], x[2], x[3], x[4], x[5], x[6], x[7]);
        inverse_affine(x);
    }
}

template <bool CALL>
__device__ __forceinline__ void sub_bytes(uint32_t (&S)[128]) {
#pragma unroll
    for (int p = 0; p < 16; p++) {
        if (!CALL) {
            sbox_circuit(S[8 * p + 0], S[8 * p + 1], S[8 * p + 2], S[8 * p + 3], S[8 * p + 4], S[8 * p + 5],
                         S[8 * p + 6], S[8 * p + 7]);
            continue;
        }
        Byte8 b{S[8 * p + 0], S[8 * p + 1], S[8 * p + 2], S[8 * p + 3],
                S[8 * p + 4], S[8 * p + 5], S[8 * p + 6], S[8 * p + 7]};
        b = sbox_call(b);
        S[8 * p + 0] = b.x0;
        S[8 * p + 1] = b.x1;
        S[8 * p + 2] = b.x2;
        S[8 * p + 3] = b.x3;
        S[8 * p + 4] = b.x4;
        S[8 * p + 5] = b.x5;
        S[8 * p + 6] = b.x6;
        S[8 * p + 7] = b.x7;
    }
}

// ShiftRows, then MixColumns (when MIX), then AddRoundKey with the plane masks
// k[0..127] (each 0 or ~0).  Output byte r + 4c takes input byte
// r + 4((c + r) mod 4); per column, with a_r those four bytes,
//   out_r = a_r ^ t ^ xtime(a_r ^ a_{r+1}),  t = a_0 ^ a_1 ^ a_2 ^ a_3,
// which is 2a_r ^ 3a_{r+1} ^ a_{r+2} ^ a_{r+3}.  xtime on planes: bit b takes
// bit b-1, and bits 1, 3, 4 also take bit 7 (x^8 = x^4 + x^3 + x + 1).
template <bool MIX>
__device__ __forceinline__ void shift_mix_key(uint32_t (&S)[128], const uint32_t* k) {
    uint32_t N[128];
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const int src[4] = {0 + 4 * ((c + 0) & 3), 1 + 4 * ((c + 1) & 3), 2 + 4 * ((c + 2) & 3),
                            3 + 4 * ((c + 3) & 3)};
        if constexpr (!MIX) {
#pragma unroll
            for (int r = 0; r < 4; r++)
#pragma unroll
                for (int b = 0; b < 8; b++) N[8 * (r + 4 * c) + b] = S[8 * src[r] + b] ^ k[8 * (r + 4 * c) + b];
            continue;
        }
        uint32_t t[8];
#pragma unroll
        for (int b = 0; b < 8; b++)
            t[b] = S[8 * src[0] + b] ^ S[8 * src[1] + b] ^ S[8 * src[2] + b] ^ S[8 * src[3] + b];
#pragma unroll
        for (int r = 0; r < 4; r++) {
            uint32_t u[8];
#pragma unroll
            for (int b = 0; b < 8; b++) u[b] = S[8 * src[r] + b] ^ S[8 * src[(r + 1) & 3] + b];
            uint32_t x2[8];
            x2[0] = u[7];
            x2[1] = u[0] ^ u[7];
            x2[2] = u[1];
            x2[3] = u[2] ^ u[7];
            x2[4] = u[3] ^ u[7];
            x2[5] = u[4];
            x2[6] = u[5];
            x2[7] = u[6];
#pragma unroll
            for (int b = 0; b < 8; b++)
                N[8 * (r + 4 * c) + b] = S[8 * src[r] + b] ^ t[b] ^ x2[b] ^ k[8 * (r + 4 * c) + b];
        }
    }
#pragma unroll
    for (int i = 0; i < 128; i++) S[i] = N[i];
}

// u times x on planes.
__device__ __forceinline__ void xtime_planes(const uint32_t* u, uint32_t* y) {
    y[0] = u[7];
    y[1] = u[0] ^ u[7];
    y[2] = u[1];
    y[3] = u[2] ^ u[7];
    y[4] = u[3] ^ u[7];
    y[5] = u[4];
    y[6] = u[5];
    y[7] = u[6];
}

// InvShiftRows, then InvMixColumns (when MIX) and AddRoundKey: the order of the
// equivalent inverse cipher.  InvMixColumns is MixColumns after
// a_r ^= x^2 (a_r ^ a_{r+2}).
template <bool MIX>
__device__ __forceinline__ void inv_shift_mix_key(uint32_t (&S)[128], const uint32_t* k) {
    uint32_t N[128];
#pragma unroll
    for (int c = 0; c < 4; c++) {
        uint32_t a[4][8];
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int b = 0; b < 8; b++) a[r][b] = S[8 * (r + 4 * ((c - r) & 3)) + b];
        if constexpr (MIX) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                uint32_t v[8], x1[8], x2[8];
#pragma unroll
                for (int b = 0; b < 8; b++) v[b] = a[h][b] ^ a[h + 2][b];
                xtime_planes(v, x1);
                xtime_planes(x1, x2);
#pragma unroll
                for (int b = 0; b < 8; b++) {
                    a[h][b] ^= x2[b];
                    a[h + 2][b] ^= x2[b];
                }
            }
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            uint32_t x2[8];
            if constexpr (MIX) {
                uint32_t u[8];
#pragma unroll
                for (int b = 0; b < 8; b++) u[b] = a[r][b] ^ a[(r + 1) & 3][b];
                xtime_planes(u, x2);
            }
#pragma unroll
            for (int b = 0; b < 8; b++) {
                const uint32_t kb = k[8 * (r + 4 * c) + b];
                if constexpr (MIX)
                    N[8 * (r + 4 * c) + b] =
                        x2[b] ^ a[(r + 1) & 3][b] ^ (a[(r + 2) & 3][b] ^ a[(r + 3) & 3][b]) ^ kb;
                else
                    N[8 * (r + 4 * c) + b] = a[r][b] ^ kb;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 128; i++) S[i] = N[i];
}

// The forward cipher on planes; km holds (NR + 1) x 128 round-key masks, in
// shared memory or in the parameter bank.  CALL: the S-box as a function.  The round loop is not unrolled: one round is ~2,000
// instructions, and 14 unrolled rounds would not fit the instruction cache.
// The final round (no MixColumns) stays inside the loop behind a uniform
// branch: as a separate copy after the loop, its state assignment differed
// from the loop's and the kernel spilled ~0.9 KB per thread.
template <int NR, bool CALL>
__device__ __forceinline__ void bs_encrypt(uint32_t (&S)[128], const uint32_t* km) {
#pragma unroll
    for (int i = 0; i < 128; i++) S[i] ^= km[i];
#pragma unroll 1
    for (int r = 1; r <= NR; r++) {
        sub_bytes<CALL>(S);
        if (r < NR)
            shift_mix_key<true>(S, km + 128 * r);
        else
            shift_mix_key<false>(S, km + 128 * r);
    }
}

// The equivalent inverse cipher (FIPS-197 section 5.3.5) on planes; km holds the
// masks of its schedule.
template <int NR>
__device__ __forceinline__ void bs_decrypt(uint32_t (&S)[128], const uint32_t* km) {
#pragma unroll
    for (int i = 0; i < 128; i++) S[i] ^= km[i];
#pragma unroll 1
    for (int r = 1; r <= NR; r++) {
        inv_sub_bytes(S);
        if (r < NR)
            inv_shift_mix_key<true>(S, km + 128 * r);
        else
            inv_shift_mix_key<false>(S, km + 128 * r);
    }
}

}  // namespace dev
}  // namespace kgpu
