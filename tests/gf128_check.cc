// The long tweak jump (kgpu::dev::gf128_jump), on the CPU.  Reads lines
// "w0 w1 w2 w3 j" (words in hex, little-endian; j decimal); prints the words
// of T * x^j.
#include <cstdio>

#include "gf128_jump.cuh"

int main() {
    unsigned w[4], j;
    while (std::scanf("%x %x %x %x %u", &w[0], &w[1], &w[2], &w[3], &j) == 5) {
        uint32_t a = w[0], b = w[1], c = w[2], d = w[3];
        kgpu::dev::gf128_jump(a, b, c, d, j);
        std::printf("%08x %08x %08x %08x\n", a, b, c, d);
    }
    return 0;
}
