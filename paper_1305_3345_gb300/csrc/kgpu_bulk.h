// Parameter blocks and launch entry points of the bulk kernels (kgpu_bulk.cu):
// one kernel per mode, direction and key size, for the per-call transforms.
// Kept apart from the batched and serving formats so that the bulk kernels'
// sources are exactly aes_device.cuh, bitslice_device.cuh, gf128_jump.cuh,
// sbox_circuit.cuh, kgpu_bulk.cu and this header.
#pragma once
#include <cuda.h>  // CUtensorMap
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace kgpu {

constexpr int kMaxRoundKeyWords = 60;  // AES-256: 4 * (14 + 1)

// Shared-memory footprint of the table layouts (see aes_device.cuh).
constexpr size_t kRegionBytes = 65536;
constexpr size_t kSmemEnc = 2 * kRegionBytes;  // regions A, B
constexpr size_t kSmemDec = 3 * kRegionBytes;  // regions A, B, C

// Threads per CTA of the bulk kernels (one CTA per SM).
constexpr int kBulkThreads = 1024;

// Large calls on tables and bit-planes at once (mixed_kernel, mixed_cbc_dec_kernel):
// 16 warps make table lookups and 4 run the bitsliced cipher.  The CTA is
// launched with 96 registers a thread, which setmaxnreg hands out again as 64
// and 224; the shares may not exceed what the launch has, or the warps that
// ask for more would wait for ever.
constexpr int kMixTableWarps = 16, kMixPlaneWarps = 4;
constexpr int kMixThreads = (kMixTableWarps + kMixPlaneWarps) * 32;
constexpr int kMixLaunchRegs = 96, kMixTableRegs = 64, kMixPlaneRegs = 224;
static_assert(kMixTableWarps * kMixTableRegs + kMixPlaneWarps * kMixPlaneRegs <=
                  (kMixTableWarps + kMixPlaneWarps) * kMixLaunchRegs,
              "register shares exceed the launch's registers");
static_assert(kMixTableWarps % 4 == 0 && kMixPlaneWarps % 4 == 0, "setmaxnreg acts on whole warpgroups");
constexpr uint32_t kMixSpanChunks = 32;  // a bitsliced span in 32-block chunks
constexpr size_t kMixTweakBytes = (kMixTableWarps + kMixPlaneWarps) * 512;  // E_K2 of 32 units per warp

// CBC encryption with a chain split over 2 or 4 lanes: at most 16 warps per CTA.
constexpr int kCbcSplitThreads = 512;

// XTS with ciphertext stealing: 24 warps (80 registers a thread, for the two
// words of an unaligned block in flight), two 16-byte words per thread after
// the tables.
constexpr int kCtsThreads = 768;
static_assert(kSmemDec + kCtsThreads * 32 <= 232448, "ciphertext stealing exceeds the 227-KB shared-memory limit");

// Staged CBC encryption: up to 20 warps per CTA (96 registers a thread), each
// with a 32-page x 8-block staging area (4608 B) after the two table regions.
// The launch picks the warp count for the page count (cbc_enc_staged_warps).
constexpr int kCbcEncStagedMaxWarps = 20;
constexpr int kCbcEncStagedThreads = kCbcEncStagedMaxWarps * 32;
constexpr size_t kStageWarpSmem = 4608;
constexpr size_t kSmemEncStaged = kSmemEnc + kCbcEncStagedMaxWarps * kStageWarpSmem;
static_assert(kSmemEncStaged <= 232448, "staged CBC encryption exceeds the 227-KB shared-memory limit");

// Warps per CTA of the staged CBC-encryption launch for `groups` groups of 32
// pages on num_sms SMs (one CTA per SM).
int cbc_enc_staged_warps(uint64_t groups, int num_sms);

// CBC encryption staged by the tensor-memory-access engine: each warp moves 8
// blocks of its 32 pages at a time as one 2-D tile (32 pages x 128 B, 128-byte
// swizzle) into a 4-KiB buffer after the table regions, with an mbarrier per
// warp after the buffers.
constexpr size_t kTmaWarpBytes = 4096;
constexpr size_t kSmemEncTma = kSmemEnc + kCbcEncStagedMaxWarps * (kTmaWarpBytes + 8);
static_assert(kSmemEncTma <= 232448, "TMA-staged CBC encryption exceeds the 227-KB shared-memory limit");

// Where dynamic shared memory starts in a CTA's shared window (the reserved
// system area comes first); the kernels fold it into their load offsets.
constexpr int kSmemReservedBytes = 1024;

// Parameters of the bulk XTS / ECB kernels (passed by value, read from the
// constant bank).
struct BulkParams {
    const uint4* src;
    uint4* dst;
    uint64_t nblocks;       // 16-byte blocks in the buffer
    uint32_t bps;           // blocks per data unit (XTS)
    uint32_t cta_rest;      // set by the launch: CTA b has cta_chunks 32-block chunks,
    uint32_t cta_chunks;    // one more if b < cta_rest
    uint32_t link;          // 1: pages cross the host link, which bounds the call
    uint64_t first_sector;  // number of the first data unit (XTS)
    uint32_t rk[kMaxRoundKeyWords];  // data key schedule (encryption or decryption order)
    uint32_t tk[kMaxRoundKeyWords];  // tweak key schedule (always encryption)
};

// Parameters of the mixed kernel: the same, the spans that each bitsliced warp
// takes from the start of its CTA's run, and the data key's plane masks (bit i
// of round key r as 0 or ~0 at 128 r + i).
struct MixParams {
    BulkParams b;
    uint32_t spans;
    alignas(16) uint32_t masks[15 * 128];
};

// Parameters of the CBC kernels.
struct CbcParams {
    const uint4* src;
    uint4* dst;
    const uint4* ivs;       // one per page
    uint64_t npages;
    uint32_t bpp;           // blocks per page
    uint32_t cta_rest;      // set by the decryption launch: CTA b has cta_items pages or
    uint32_t cta_items;     // chunks, one more if b < cta_rest
    uint32_t link;          // 1: pages cross the host link
    uint32_t rk[kMaxRoundKeyWords];
};

// Parameters of the TMA-staged CBC encryption: the source and destination as
// 2-D tensors of 32-bit words (page words x pages, page stride bpp * 16 bytes)
// read and written in 32 x 32 boxes.
struct CbcTmaParams {
    CUtensorMap src_map;
    CUtensorMap dst_map;
    const uint4* ivs;  // one per page
    uint64_t npages;
    uint32_t bpp;      // blocks per page, a multiple of 8
    uint32_t pad0;
    uint32_t rk[kMaxRoundKeyWords];
};

struct MixCbcParams {
    CbcParams c;
    uint32_t spans;
    alignas(16) uint32_t masks[15 * 128];
};

// XTS with ciphertext stealing: data units of du bytes, du >= 16 and not a
// multiple of 16 (IEEE 1619-2007 5.3.2 / 5.4.2).  Unit u starts at byte u * du.
struct CtsParams {
    const uint8_t* src;
    uint8_t* dst;
    uint64_t units;
    uint64_t du;
    uint64_t first_sector;
    uint64_t cta_units;  // set by the launch: CTA b has cta_units units, one more if b < cta_rest
    uint32_t cta_rest;
    uint32_t pad0;
    uint32_t rk[kMaxRoundKeyWords];
    uint32_t tk[kMaxRoundKeyWords];
};

// ---------------------------------------------------------------------------
// Which form a call takes, from its sizes alone.
// ---------------------------------------------------------------------------

// Spans that each bitsliced warp of a CTA takes from a run of cta_chunks
// 32-block chunks; 0: the call stays on the tables.  A warp that takes one span
// too many costs the call up to a span's time, so a span is given for every
// so many chunks as the table warps encipher meanwhile, rounded down.  1 GiB
// (13,797 chunks a CTA) of AES-256-XTS by spans per warp: 0 1,584 us, 10 1,475,
// 11 1,527; of AES-128 0 1,155, 9 1,099, 10 1,160; of ECB, which forms no
// tweaks, with AES-256 0 1,573, 10 1,443, 11 1,428, with AES-128 9 1,066, 11
// 1,046; of decryption with AES-256-XTS 0 1,591, 8 1,524, 9 1,540, with AES-128
// 0 1,165, 7 1,130, 8 1,135; of CBC decryption with AES-256 0 1,616, 10 1,541, 11
// 1,563, with AES-128 0 1,189, 10 1,121, 11 1,165.  Units under 512 bytes have
// more tweaks than a span has lanes, and pages that cross the host link are
// bound by it.
inline uint32_t mix_spans(uint32_t cta_chunks, int nr, int dir, bool tweak, uint32_t unit_blocks, bool link) {
    if (link || unit_blocks < 32 || (tweak && nr == 12)) return 0;
    const bool big = nr == 14;
    uint32_t per_span;
    if (dir == 0) per_span = tweak ? (big ? 1300 : 1400) : (big ? 1200 : 1250);
    else per_span = tweak ? (big ? 1600 : 1800) : 1300;
    return cta_chunks / per_span;
}

constexpr uint32_t kLineBlocks = 8;  // blocks in a 128-byte line

// Lanes that share a page's chain in CBC encryption.  Few pages are a chain's
// latency, which two or four lanes per page shorten; many are the lookups'
// rate, which one lane per page uses best.  4-KiB pages, AES-128, one / two /
// four lanes: 8 pages per SM 145 / 107 / 103 us, 32 pages 145 / 109 / 107, 64
// pages 147 / 121 / 121, 128 pages 153 / 152 / 180, 160 pages 206 / 182 / 288,
// 192 pages 208 / 207 / 295, 224 pages 215 / 248 / 316.  Pages that cannot be
// staged cross later (4112 B, AES-256: 224 pages 299 / 286, 256 pages 306 / 309).
//
// Shared lanes move 16 bytes a page at a time.  Over the host link that wins
// only for a few pages; from there whole lines, which one lane per page moves
// staged, are several times as fast.  kgpu_crypt on registered 4-KiB pages,
// shared / staged lanes: AES-128 8 pages 142 / 159 us, 64 pages 144-163 / 159,
// 1,024 pages 288 / 160, 16,384 pages 1,984 / 510; AES-192 128 pages 172 / 182,
// 384 pages 192 / 183; AES-256 256 pages 182 / 206, 1,024 pages 288 / 208.
inline int cbc_enc_lanes(uint64_t npages, uint32_t bpp, int nr, uint64_t sms, bool link) {
    const bool lines = bpp % kLineBlocks == 0;
    if (link && lines && npages > (nr == 10 ? 32u : nr == 12 ? 128u : 256u)) return 1;
    if (npages <= 32 * sms) return 4;
    return npages <= (lines ? 192 : 240) * sms ? 2 : 1;
}

// CTAs for teams of one warp each that split chains over lanes.  Two warps share
// an SM before the next is taken, which costs a chain nothing; past an eighth
// of the SMs three do, so that calls on several streams run beside each other
// (4 MiB of AES-128 on eight streams: two warps an SM 47.7 us a call, three
// 33.4, a warp a page group without split chains 32.8).  A call by itself takes
// 102.3 us with three, 101.7 with two and 103.7 with four.
inline uint64_t cbc_enc_split_ctas(uint64_t teams, uint64_t sms) {
    const uint64_t two = (teams + 1) / 2, three = (teams + 2) / 3;
    const uint64_t eighth = sms / 8;
    const uint64_t n = two <= eighth ? two : three > eighth ? three : eighth;
    return n < 1 ? 1 : n < sms ? n : sms;
}

// SMs for a launch whose pages cross the host link.  A quarter of them enciphers
// about as fast as the link moves pages in both directions (171 GB/s), leaves
// the others free and, for short calls, is the faster: AES-256-XTS in 4-KiB units
// on 38 / 114 / 152 SMs 4 MiB 54 / 59 / 61 us, 16 MiB 130 / 136 / 138, 64 MiB 434
// / 439 / 442.  Long calls run into the lookups there, the sooner the more of
// them go to tweaks, and want three quarters: 128 MiB 844 / 843 / 852, 1 GiB 6,604
// / 6,516 / 6,566; 512-byte units 32 MiB 240 / 236 / 240, 64 MiB 455 / 438 / 444, 1
// GiB 6,831 / 6,533 / 6,576.  (Half the SMs are slower than either at 4-KiB units,
// 7,090 at 1 GiB, in every run; why is not known.)  Units of less than 512 bytes
// keep the whole device.
inline int link_sms(int num_sms, uint32_t unit_blocks, uint64_t bytes) {
    if (unit_blocks < 32) return num_sms;
    const uint64_t most = (unit_blocks >= 128 ? 96ull : 48ull) << 20;
    return bytes <= most ? (num_sms + 3) / 4 : (3 * num_sms + 3) / 4;
}

// SMs for CBC decryption: over the host link, from the sizes where a call that
// takes them all is bound by it, as for XTS (registered 4-KiB pages, AES-128, 152
// / 38 SMs: 1 MiB 24.5 / 24.3 us, AES-256 24.6 / 25.9; 2 MiB 34.4 / 31.6; 4 MiB
// 50.8 / 44.8; 8 MiB 77.3 / 71.2).
inline int cbc_dec_sms(int num_sms, uint32_t bpp, uint64_t bytes, bool link) {
    return link && bytes >= (2ull << 20) ? link_sms(num_sms, bpp, bytes) : num_sms;
}

cudaError_t launch_xts(const BulkParams& p, int nr, int dir, int num_sms, cudaStream_t s);
cudaError_t launch_xts_cts(const CtsParams& p, int nr, int dir, int num_sms, cudaStream_t s);
cudaError_t launch_ecb(const BulkParams& p, int nr, int dir, int num_sms, cudaStream_t s);
cudaError_t launch_cbc_dec(const CbcParams& p, int nr, int num_sms, cudaStream_t s);
cudaError_t launch_cbc_enc(const CbcParams& p, int nr, int num_sms, cudaStream_t s);
cudaError_t upload_tables(const uint32_t* te0, const uint32_t* td0, const uint32_t* isb4);
// Bounded waits of the bulk kernels that ran out on the current device (a
// process-wide count; 0 unless a tensor copy never completed).
cudaError_t bulk_wait_timeouts(unsigned int* out);
cudaError_t configure_kernels();  // opt-in to large dynamic shared memory

}  // namespace kgpu
