// Launch decisions for batched and served requests (kgpu::hostutil), on the
// CPU.  Reads lines
//   "b chunks nblocks burst_bytes workers host max_tiles" -> prints burst_tile_chunks
//   "r ctas sms"                -> prints resident_ctas
//   "t ctas sms warps n" then n lengths in bytes -> prints default_tile_chunks for
//                                  the launch's resident warps
//   "p ctas sms warps n" then n lines "mode nblocks unit_blocks tile_units flags"
//                               -> prints plan_batch's header (total_tiles long_tiles
//                                  long_warps ctas), the run order, the tile prefix,
//                                  and each request's flags and tile_units
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
        } else if (kind[0] == 'r') {
            unsigned ctas;
            int sms;
            if (std::scanf("%u %d", &ctas, &sms) != 2) return 2;
            std::printf("%u\n", kgpu::hostutil::resident_ctas(ctas, sms));
        } else if (kind[0] == 't') {
            unsigned ctas, warps, n;
            int sms;
            if (std::scanf("%u %d %u %u", &ctas, &sms, &warps, &n) != 4) return 2;
            std::vector<kgpu_request> r(n);
            for (auto& q : r) {
                unsigned long long len;
                if (std::scanf("%llu", &len) != 1) return 2;
                q.len = len;
            }
            const uint64_t at_once = (uint64_t)kgpu::hostutil::resident_ctas(ctas, sms) * warps;
            std::printf("%u\n", kgpu::hostutil::default_tile_chunks(r.data(), n, at_once));
        } else if (kind[0] == 'p') {
            unsigned ctas, warps, n;
            int sms;
            if (std::scanf("%u %d %u %u", &ctas, &sms, &warps, &n) != 4) return 2;
            std::vector<uint64_t> words(kgpu::batch_bytes(n) / 8 + 1);
            uint8_t* buf = reinterpret_cast<uint8_t*>(words.data());
            auto* d = reinterpret_cast<kgpu::ReqDesc*>(buf + kgpu::batch_desc_offset());
            for (unsigned i = 0; i < n; i++) {
                unsigned long long nb;
                d[i] = kgpu::ReqDesc{};
                if (std::scanf("%u %llu %u %u %u", &d[i].mode, &nb, &d[i].unit_blocks, &d[i].tile_units, &d[i].flags) != 5)
                    return 2;
                d[i].nblocks = nb;
            }
            kgpu::hostutil::plan_batch(buf, n, [&](uint32_t i) { return d[i].nblocks == 0; },
                                       kgpu::hostutil::resident_ctas(ctas, sms), warps);
            const auto* h = reinterpret_cast<const kgpu::BatchHeader*>(buf);
            const auto* prefix = reinterpret_cast<const uint64_t*>(buf + kgpu::batch_prefix_offset(n));
            const auto* order = reinterpret_cast<const uint32_t*>(buf + kgpu::batch_order_offset(n));
            std::printf("%llu %llu %u %u\n", (unsigned long long)h->total_tiles, (unsigned long long)h->long_tiles,
                        h->long_warps, h->ctas);
            for (unsigned i = 0; i < n; i++) std::printf("%u ", order[i]);
            std::printf("\n");
            for (unsigned i = 0; i <= n; i++) std::printf("%llu ", (unsigned long long)prefix[i]);
            std::printf("\n");
            for (unsigned i = 0; i < n; i++) std::printf("%u %u ", d[i].flags, d[i].tile_units);
            std::printf("\n");
        } else {
            return 2;
        }
    }
    return 0;
}
