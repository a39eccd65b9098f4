// Launch decisions for batched and served requests (kgpu::hostutil), on the
// CPU.  Reads lines
//   "b chunks nblocks burst_bytes workers host max_tiles" -> prints burst_tile_chunks
#include <cstdio>
#include <vector>

#include "kgpu_ctx.h"

int main() {
    char kind[2];
    while (std::scanf("%1s", kind) == 1) {
        if (kind[0] == 'b') {
            unsigned chunks;
            unsigned long long nblocks, burst, workers, most;
            int host;
            if (std::scanf("%u %llu %llu %llu %d %llu", &chunks, &nblocks, &burst, &workers, &host, &most) != 6) return 2;
            std::printf("%u\n", kgpu::hostutil::burst_tile_chunks(chunks, nblocks, burst, workers, host != 0, most));
        } else {
            return 2;
        }
    }
    return 0;
}
