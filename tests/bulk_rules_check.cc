// The launch rules of the bulk kernels (kgpu_bulk.h), on the CPU.  Reads lines
//   "e npages bpp nr sms link" -> prints cbc_enc_lanes
//   "s teams sms"               -> prints cbc_enc_split_ctas
//   "l sms unit_blocks bytes"   -> prints link_sms
//   "d sms bpp bytes link"      -> prints cbc_dec_sms
//   "m cta_chunks nr dir tweak unit_blocks link" -> prints mix_spans
#include <cstdio>

#include "kgpu_bulk.h"

int main() {
    char kind[2];
    while (std::scanf("%1s", kind) == 1) {
        if (kind[0] == 'e') {
            unsigned long long npages, sms;
            unsigned bpp;
            int nr, link;
            if (std::scanf("%llu %u %d %llu %d", &npages, &bpp, &nr, &sms, &link) != 5) return 2;
            std::printf("%d\n", kgpu::cbc_enc_lanes(npages, bpp, nr, sms, link != 0));
        } else if (kind[0] == 's') {
            unsigned long long teams, sms;
            if (std::scanf("%llu %llu", &teams, &sms) != 2) return 2;
            std::printf("%llu\n", (unsigned long long)kgpu::cbc_enc_split_ctas(teams, sms));
        } else if (kind[0] == 'l') {
            int sms;
            unsigned unit;
            unsigned long long bytes;
            if (std::scanf("%d %u %llu", &sms, &unit, &bytes) != 3) return 2;
            std::printf("%d\n", kgpu::link_sms(sms, unit, bytes));
        } else if (kind[0] == 'd') {
            int sms, link;
            unsigned bpp;
            unsigned long long bytes;
            if (std::scanf("%d %u %llu %d", &sms, &bpp, &bytes, &link) != 4) return 2;
            std::printf("%d\n", kgpu::cbc_dec_sms(sms, bpp, bytes, link != 0));
        } else if (kind[0] == 'm') {
            unsigned chunks, unit;
            int nr, dir, tweak, link;
            if (std::scanf("%u %d %d %d %u %d", &chunks, &nr, &dir, &tweak, &unit, &link) != 6) return 2;
            std::printf("%u\n", kgpu::mix_spans(chunks, nr, dir, tweak != 0, unit, link != 0));
        } else {
            return 2;
        }
    }
    return 0;
}
