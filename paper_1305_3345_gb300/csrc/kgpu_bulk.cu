// Bulk device-resident kernels: XTS (IEEE 1619), ECB, CBC decrypt (parallel
// over blocks) and CBC encrypt (parallel over pages).
//
// All share one structure: one CTA per SM fills its replicated lookup tables
// into shared memory once (see aes_device.cuh).  For XTS, ECB and CBC
// decryption every CTA owns an equal contiguous range of the buffer and its 32
// warps equal parts of that, which they walk 32 blocks (512 B) at a time, one
// 16-byte block per lane, so each warp-wide load and store is a fully
// coalesced 512-byte transaction.  CBC encryption runs one page's chain per lane, 32
// pages per warp, with the warp count set by the page count, and moves the
// pages through shared memory in whole lines (register-staged, or as tensor
// tiles for large launches).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <mutex>

#include "aes_device.cuh"
#include "kgpu_bulk.h"

namespace kgpu {

using namespace dev;

static_assert(kSmemBase == (uint32_t)kSmemReservedBytes, "table offsets assume the reserved shared area");

// Cipher constants, uploaded once per device by upload_tables().
__device__ uint32_t g_te0[256];
__device__ uint32_t g_td0[256];
__device__ uint32_t g_isb4[256];

namespace {

// Regions A/B <- T0..T3 built from base[] by byte rotation.  A row is 16
// pieces of 16 bytes, eight copies-of-four of the even table's word and eight
// of the odd table's; a thread writes one piece of region A and the same word
// turned by 16 bits to region B.  The 128 KiB then take their 1,024
// wavefronts and one round of loads.  Every launch pays for it: with one
// 4-byte store per word and a load before each it took 2.9 us of a launch
// (6,000 cycles); back-to-back 4-KiB XTS calls took 12.3 us each, 10.3 this
// way.
__device__ __forceinline__ void fill_round_tables(uint4* w, const uint32_t* base) {
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < 4096; i += blockDim.x) {
        uint32_t v = base[i >> 4];
        if (i & 8u) v = rotl8(v);
        w[i] = make_uint4(v, v, v, v);
        v = rotl16(v);
        w[4096 + i] = make_uint4(v, v, v, v);
    }
}

__device__ __forceinline__ void fill_enc(char* smem) {
    fill_round_tables(reinterpret_cast<uint4*>(smem), g_te0);
}

// Regions A/B <- Td0..Td3; region C <- InvS (first half) and, for kernels that
// form tweaks, Te0 (second half).
template <bool TWEAK>
__device__ __forceinline__ void fill_dec(char* smem) {
    uint4* w = reinterpret_cast<uint4*>(smem);
    fill_round_tables(w, g_td0);
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < (TWEAK ? 4096u : 2048u); i += blockDim.x) {
        const uint32_t x = TWEAK ? i >> 4 : i >> 3;
        const uint32_t v = TWEAK && (i & 8u) ? g_te0[x] : g_isb4[x];
        w[8192 + (TWEAK ? i : (x << 4 | (i & 7u)))] = make_uint4(v, v, v, v);
    }
}

__device__ __forceinline__ void xor4(uint4& v, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    v.x ^= a;
    v.y ^= b;
    v.z ^= c;
    v.w ^= d;
}

// a / b where a rarely needs more than 32 bits.
__device__ __forceinline__ uint64_t div_small(uint64_t a, uint32_t b) {
    return (a >> 32) == 0 ? (uint64_t)((uint32_t)a / b) : a / b;
}

// ---------------------------------------------------------------------------
// XTS (and ECB when TWEAK is false).  Bound by the shared-memory lookups (one
// wavefront a cycle); a CTA owns one contiguous run of 32-block chunks and its
// warps equal parts of it.
//
// Tweaks: the E_K2 of the data units that a group of warps is about to touch
// are enciphered first, one unit per thread, into shared memory (a phase), and
// a lane entering a unit reads its E_K2 there and multiplies by alpha^j in
// closed form; a lane staying in its unit steps its tweak by alpha^32.  The
// group is the CTA for units of at least a chunk, so that a unit is enciphered
// once per CTA and a short run costs one warp's AES: with 32 units enciphered
// by every warp for itself, 1 MiB of 4-KiB units spent as many lookups on
// tweaks as on data.  Smaller units change within a chunk; there each warp
// takes its own 32 units at a time and no barrier is needed.
// 1 MiB of 4-KiB units, AES-256 decryption, back to back on the GPU: 14.4 -> 8.2 us;
// 16 MiB of encryption 34.9 -> 30.8 us.
// ---------------------------------------------------------------------------
template <int NR, int DIR, bool TWEAK>
__global__ void __launch_bounds__(kBulkThreads, 1) bulk_kernel(const __grid_constant__ BulkParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;  // uniform over the CTA; refused at init
    if (DIR == 0) fill_enc(smem);
    else fill_dec<TWEAK>(smem);
    __syncthreads();

    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    constexpr uint32_t kWarps = kBulkThreads / 32;
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const Rep1<2> IS{lane * 4u};
    const Rep1<2> TE{lane * 4u + 128u};
    const ParamKey K{p.rk};
    const ParamKey TK{p.tk};

    // this CTA's chunks, and this warp's part of them
    const uint32_t own = p.cta_chunks + (blockIdx.x < p.cta_rest ? 1u : 0u);
    const uint64_t first = (uint64_t)p.cta_chunks * blockIdx.x + min(blockIdx.x, p.cta_rest);
    const uint32_t wa = (uint32_t)((uint64_t)own * warp / kWarps);
    const uint32_t we = (uint32_t)((uint64_t)own * (warp + 1) / kWarps);

    if constexpr (!TWEAK) {
        uint64_t blk = ((first + wa) << 5) + lane;
        // the next chunk is fetched while this one is enciphered
        uint4 nxt = wa < we && blk < p.nblocks ? p.src[blk] : make_uint4(0, 0, 0, 0);
        for (uint32_t c = wa; c < we; ++c, blk += 32) {
            uint4 v = nxt;
            if (c + 1 < we && blk + 32 < p.nblocks) nxt = p.src[blk + 32];
            if (DIR == 0) encrypt_block<NR>(v.x, v.y, v.z, v.w, T, K);
            else decrypt_block<NR>(v.x, v.y, v.z, v.w, T, IS, K);
            if (blk < p.nblocks) p.dst[blk] = v;
        }
        return;
    }

    const uint32_t bps = p.bps;
    const bool shared = bps >= 32;  // the CTA forms the tweaks together
    const uint32_t gthreads = shared ? (uint32_t)kBulkThreads : 32u;
    const uint32_t gwarp = shared ? warp : 0u, gwarps = shared ? kWarps : 1u;
    uint4* tw = reinterpret_cast<uint4*>(smem + (DIR == 0 ? kSmemEnc : kSmemDec)) + (shared ? 0u : warp * 32u);
    auto group_sync = [&]() {
        if (shared) __syncthreads();
        else __syncwarp();
    };
    uint64_t c = first + (shared ? 0u : wa);
    uint32_t left = shared ? own : we - wa;
    bool again = false;
    while (left) {
        // the phase: as many chunks as have their units among gthreads
        const uint64_t b0 = c << 5;
        const uint64_t unit0 = div_small(b0, bps);
        const uint32_t o = (uint32_t)(b0 - unit0 * bps);  // b0's place in unit0
        const uint64_t fit = ((uint64_t)gthreads * bps - o) >> 5;  // >= 1
        const uint32_t n = (uint32_t)min((uint64_t)min(left, 1u << 24), fit);
        const uint32_t a = n * gwarp / gwarps, e = n * (gwarp + 1) / gwarps;
        uint64_t blk = b0 + ((uint64_t)a << 5) + lane;
        uint4 nxt = a < e && blk < p.nblocks ? p.src[blk] : make_uint4(0, 0, 0, 0);
        if (again) group_sync();  // the last phase's tweaks have been read
        again = true;
        if ((uint64_t)gwarp * 32 * bps < (uint64_t)o + ((uint64_t)n << 5)) {  // units of this phase among this warp's
            const uint64_t unit = p.first_sector + unit0 + gwarp * 32 + lane;
            uint4 z = make_uint4((uint32_t)unit, (uint32_t)(unit >> 32), 0, 0);
            if (DIR == 0) encrypt_block<NR>(z.x, z.y, z.z, z.w, T, TK);
            else encrypt_block<NR>(z.x, z.y, z.z, z.w, TE, TK);
            tw[gwarp * 32 + lane] = z;
        }
        group_sync();
        if (a < e) {
            const uint64_t q = (uint64_t)o + ((uint64_t)a << 5) + lane;
            uint32_t u = (uint32_t)div_small(q, bps);  // unit of the phase
            uint32_t j = (uint32_t)(q - (uint64_t)u * bps);
            uint4 t = tw[u];
            gf128_mul_xpow(t.x, t.y, t.z, t.w, j);
            for (uint32_t i = a; i < e; ++i) {
                uint4 v = nxt;
                if (i + 1 < e && blk + 32 < p.nblocks) nxt = p.src[blk + 32];
                xor4(v, t.x, t.y, t.z, t.w);
                if (DIR == 0) encrypt_block<NR>(v.x, v.y, v.z, v.w, T, K);
                else decrypt_block<NR>(v.x, v.y, v.z, v.w, T, IS, K);
                xor4(v, t.x, t.y, t.z, t.w);
                if (blk < p.nblocks) p.dst[blk] = v;
                blk += 32;
                if (i + 1 < e) {
                    j += 32;
                    if (j >= bps) {
                        const uint32_t ns = shared ? 1u : j / bps;
                        u += ns;
                        j -= ns * bps;
                        t = tw[u];
                        gf128_mul_xk(t.x, t.y, t.z, t.w, j);
                    } else {
                        gf128_mul_x32(t.x, t.y, t.z, t.w);
                    }
                }
            }
        }
        c += n;
        left -= n;
    }
}

// ---------------------------------------------------------------------------
// CBC decryption, one block per lane.  P_i = D(C_i) ^ C_{i-1}: C_{i-1} comes
// from the neighbouring lane by shuffle (lane 0 takes lane 31's block of the
// previous step, and the block before the warp's range at its start), and from
// the page IV at the first block of a page.  Bound by the lookups, so the work
// is split evenly in 32-block chunks over CTAs and warps, across page
// boundaries: whole pages per warp left 16,387 pages on 4,864 warps at 4 pages
// where 3.4 would do (64 MiB, AES-128: 82.2 -> 80.8 us) and 256 pages on 8 CTAs
// (1 MiB: 27.6 -> 6.2 us, 16 MiB: 28.7 -> 24.6 us).
//
// In place, the block before a range may not be overwritten before it is
// read.  A CTA then takes whole pages, so that only its own warps' ranges
// touch, and every warp reads that block before the barrier that precedes the
// first store.
// ---------------------------------------------------------------------------
template <int NR>
__global__ void __launch_bounds__(kBulkThreads, 1) cbc_dec_kernel(const __grid_constant__ CbcParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    fill_dec<false>(smem);

    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    constexpr uint32_t kWarps = kBulkThreads / 32;
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const Rep1<2> IS{lane * 4u};
    const ParamKey K{p.rk};

    // this CTA's blocks [b0, bend): pages in place, else 32-block chunks
    const uint32_t bpp = p.bpp;
    const uint64_t item = p.src == p.dst ? bpp : 32u;
    const uint64_t first = (uint64_t)p.cta_items * blockIdx.x + min(blockIdx.x, p.cta_rest);
    const uint32_t own = p.cta_items + (blockIdx.x < p.cta_rest ? 1u : 0u);
    const uint64_t b0 = first * item;
    const uint64_t bend = min(b0 + own * item, p.npages * bpp);
    const uint32_t chunks = (uint32_t)((bend - b0 + 31) >> 5);
    const uint32_t a = (uint32_t)((uint64_t)chunks * warp / kWarps);
    const uint32_t e = (uint32_t)((uint64_t)chunks * (warp + 1) / kWarps);
    uint64_t blk = b0 + ((uint64_t)a << 5) + lane;
    uint64_t page = div_small(blk, bpp);
    uint32_t j = (uint32_t)(blk - page * bpp);
    const bool some = a < e && blk < bend;
    uint4 carry = some && lane == 0 && j ? p.src[blk - 1] : make_uint4(0, 0, 0, 0);
    uint4 nxt = some ? p.src[blk] : make_uint4(0, 0, 0, 0);
    __syncthreads();  // the tables are filled and every carry is read

    for (uint32_t i = a; i < e; ++i) {
        const bool valid = blk < bend;
        const uint4 c = nxt;
        if (i + 1 < e && blk + 32 < bend) nxt = p.src[blk + 32];  // prefetch the next step
        // one rotation gives lane i the block of lane i-1; lane 0 receives
        // lane 31's, which it keeps for the next step and replaces by the
        // one it kept from the previous step
        const uint32_t from = (lane + 31) & 31;
        uint4 prev;
        prev.x = __shfl_sync(0xffffffffu, c.x, from);
        prev.y = __shfl_sync(0xffffffffu, c.y, from);
        prev.z = __shfl_sync(0xffffffffu, c.z, from);
        prev.w = __shfl_sync(0xffffffffu, c.w, from);
        if (lane == 0) {
            const uint4 last = prev;
            prev = carry;
            carry = last;
        }
        if (valid && j == 0) prev = p.ivs[page];
        uint4 v = c;
        decrypt_block<NR>(v.x, v.y, v.z, v.w, T, IS, K);
        xor4(v, prev.x, prev.y, prev.z, prev.w);
        if (valid) p.dst[blk] = v;
        blk += 32;
        j += 32;
        if (j >= bpp) {
            uint32_t ns = j / bpp;
            page += ns;
            j -= ns * bpp;
        }
    }
}

// ---------------------------------------------------------------------------
// CBC encryption, one page per lane: C_i = E(P_i ^ C_{i-1}) is a sequential
// chain inside a page, so parallelism comes from pages.  Warps take groups of
// 32 pages; the next plaintext block is fetched while the current one is
// encrypted.
// ---------------------------------------------------------------------------
template <int NR>
__global__ void __launch_bounds__(kBulkThreads, 1) cbc_enc_kernel(const __grid_constant__ CbcParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    fill_enc(smem);
    __syncthreads();

    const uint32_t lane = lane_id();
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const ParamKey K{p.rk};
    const uint32_t bpp = p.bpp;
    const uint64_t ngroups = (p.npages + 31) >> 5;

    for (uint64_t g = interleaved_warp(); g < ngroups; g += total_warps()) {
        // lanes without a page step along with the others, loads and stores
        // predicated off, so the warp stays converged through the chain
        const uint64_t page = (g << 5) + lane;
        const bool valid = page < p.npages;
        const uint4* in = p.src + (valid ? page : 0) * bpp;
        uint4* out = p.dst + (valid ? page : 0) * bpp;
        const uint4 z = make_uint4(0, 0, 0, 0);
        uint4 x = valid ? p.ivs[page] : z;
        // the chain is sequential, so plaintext is fetched four blocks ahead
        uint4 q0 = valid ? in[0] : z;
        uint4 q1 = valid && bpp > 1 ? in[1] : z;
        uint4 q2 = valid && bpp > 2 ? in[2] : z;
        uint4 q3 = valid && bpp > 3 ? in[3] : z;
        for (uint32_t i = 0; i < bpp; ++i) {
            const uint4 cur = q0;
            q0 = q1;
            q1 = q2;
            q2 = q3;
            if (valid && i + 4 < bpp) q3 = in[i + 4];
            xor4(x, cur.x, cur.y, cur.z, cur.w);
            encrypt_block<NR>(x.x, x.y, x.z, x.w, T, K);
            if (valid) out[i] = x;
        }
    }
}


// ---------------------------------------------------------------------------
// CBC encryption with a page's chain split over LANES = 4 or 2 lanes, for
// calls whose time is a chain's latency.  A lane holds one or two columns of
// its page's state; each round it takes the others from its neighbours by
// shuffle and makes 4 or 8 lookups of its own, with its columns of the round
// keys in registers.  A lane that holds a whole page makes 16 lookups in a row
// before the next round can start: 107 cycles a round, against 77 with four
// lanes and 78 with two.  Per round, four lanes spend 7 operations of the
// shared-memory path on 8 pages and two spend 10 on 16, where one lane per
// page spends 16 on 32: each form loses once that path is the bound (see
// launch_cbc_enc).
// ---------------------------------------------------------------------------
template <int NR, int LANES>
__global__ void __launch_bounds__(kCbcSplitThreads, 1) cbc_enc_split_kernel(const __grid_constant__ CbcParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    fill_enc(smem);
    constexpr int kCols = 4 / LANES;              // columns per lane
    constexpr uint32_t kPages = 32 / LANES;       // pages per warp
    using Piece = std::conditional_t<kCols == 1, uint32_t, uint2>;
    const uint32_t lane = lane_id();
    const uint32_t c = lane & (LANES - 1u), team = lane & ~(LANES - 1u);
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    uint32_t k[NR + 1][kCols];
#pragma unroll
    for (int r = 0; r <= NR; r++)
#pragma unroll
        for (int i = 0; i < kCols; i++) k[r][i] = p.rk[4 * r + kCols * c + i];
    const uint32_t bpp = p.bpp;
    const uint64_t ngroups = (p.npages + kPages - 1) / kPages;
    __syncthreads();

    for (uint64_t g = interleaved_warp(); g < ngroups; g += total_warps()) {
        // lanes without a page step along, loads and stores predicated off
        const uint64_t page = g * kPages + lane / LANES;
        const bool valid = page < p.npages;
        const uint64_t at = (valid ? page : 0) * bpp * LANES + c;  // in pieces
        const Piece* in = reinterpret_cast<const Piece*>(p.src) + at;
        Piece* out = reinterpret_cast<Piece*>(p.dst) + at;
        uint32_t s[4];  // this lane's columns, then the next lanes'
        auto fetch = [&](const Piece* from, bool ok, uint32_t (&v)[kCols]) {
            Piece w{};
            if (ok) w = *from;
            if constexpr (kCols == 1) {
                v[0] = w;
            } else {
                v[0] = w.x;
                v[1] = w.y;
            }
        };
        uint32_t x[kCols], q[4][kCols];
        fetch(reinterpret_cast<const Piece*>(p.ivs) + (valid ? page : 0) * LANES + c, valid, x);
        // the chain is sequential, so plaintext is fetched four blocks ahead
#pragma unroll
        for (uint32_t i = 0; i < 4; i++) fetch(in + (size_t)LANES * i, valid && i < bpp, q[i]);
        for (uint32_t i = 0; i < bpp; ++i) {
#pragma unroll
            for (int h = 0; h < kCols; h++) {
                s[h] = x[h] ^ q[0][h] ^ k[0][h];
                q[0][h] = q[1][h];
                q[1][h] = q[2][h];
                q[2][h] = q[3][h];
            }
            fetch(in + (size_t)LANES * (i + 4), valid && i + 4 < bpp, q[3]);
#pragma unroll
            for (int r = 1; r <= NR; r++) {
#pragma unroll
                for (int h = kCols; h < 4; h++)
                    s[h] = __shfl_sync(0xffffffffu, s[h % kCols], team | ((c + h / kCols) & (LANES - 1u)));
#pragma unroll
                for (int h = 0; h < kCols; h++) {
                    const uint32_t s0 = s[h], s1 = s[h + 1], s2 = s[(h + 2) & 3], s3 = s[(h + 3) & 3];
                    if (r < NR)
                        x[h] = T.t<0, 0>(s0) ^ k[r][h] ^ T.t<1, 1>(s1) ^ T.t<2, 2>(s2) ^ T.t<3, 3>(s3);
                    else  // S(x) from the byte of table (r+3)%4 that holds it unscaled
                        x[h] = merge_bytes(T.t<3, 0>(s0), T.t<0, 1>(s1), T.t<1, 2>(s2), T.t<2, 3>(s3)) ^ k[r][h];
                }
#pragma unroll
                for (int h = 0; h < kCols; h++) s[h] = x[h];
            }
            if (valid) {
                if constexpr (kCols == 1) out[(size_t)LANES * i] = x[0];
                else out[(size_t)LANES * i] = make_uint2(x[0], x[1]);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// CBC encryption, staged.  The chains are the same (one page per lane), but a
// lane's loads and stores at 4-KiB strides would touch 32 cache lines per
// warp instruction; instead each warp moves 8 blocks of each of its 32 pages at
// a time between global memory and a padded shared-memory area with
// coalesced accesses (four 128-B lines per instruction), and the lanes read
// and write their own chains there.  Used when a page is a multiple of 8
// blocks (128 B).  The next 8 blocks are fetched into registers while the
// current ones are enciphered.
// ---------------------------------------------------------------------------
constexpr int kStageBlocks = 8;
constexpr int kStageRow = kStageBlocks * 16 + 16;  // one page's 8 blocks, padded against bank conflicts
constexpr int kStageWarpBytes = 32 * kStageRow;
static_assert(kStageWarpBytes == kStageWarpSmem, "staging area size");

template <int NR>
__global__ void __launch_bounds__(kCbcEncStagedThreads, 1) cbc_enc_staged_kernel(const __grid_constant__ CbcParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    fill_enc(smem);
    __syncthreads();

    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const ParamKey K{p.rk};
    const uint32_t bpp = p.bpp;
    const uint32_t nchunks = bpp / kStageBlocks;
    char* stage = smem + kSmemEnc + warp * kStageWarpBytes;
    char* own = stage + lane * kStageRow;            // this lane's chain
    const uint32_t cp_page = lane >> 3, cp_blk = lane & 7;  // coalesced copy position
    const uint64_t ngroups = (p.npages + 31) >> 5;

    for (uint64_t g = interleaved_warp(); g < ngroups; g += total_warps()) {
        const uint64_t page = (g << 5) + lane;
        const bool valid = page < p.npages;
        uint4 x = valid ? p.ivs[page] : make_uint4(0, 0, 0, 0);
        uint4 R[4 * 2];
        auto fetch = [&](uint32_t c) {
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const uint64_t pg = (g << 5) + q * 4 + cp_page;
                R[q] = pg < p.npages ? p.src[pg * bpp + c * kStageBlocks + cp_blk] : make_uint4(0, 0, 0, 0);
            }
        };
        fetch(0);
        for (uint32_t c = 0; c < nchunks; ++c) {
            __syncwarp();  // the previous chunk's ciphertext has been written out
#pragma unroll
            for (int q = 0; q < 8; q++)
                *reinterpret_cast<uint4*>(stage + (q * 4 + cp_page) * kStageRow + cp_blk * 16) = R[q];
            __syncwarp();
            if (c + 1 < nchunks) fetch(c + 1);
#pragma unroll 1
            for (int i = 0; i < kStageBlocks; i++) {
                const uint4 pt = *reinterpret_cast<const uint4*>(own + i * 16);
                xor4(x, pt.x, pt.y, pt.z, pt.w);
                encrypt_block<NR>(x.x, x.y, x.z, x.w, T, K);
                *reinterpret_cast<uint4*>(own + i * 16) = x;
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const uint64_t pg = (g << 5) + q * 4 + cp_page;
                if (pg < p.npages)
                    p.dst[pg * bpp + c * kStageBlocks + cp_blk] =
                        *reinterpret_cast<const uint4*>(stage + (q * 4 + cp_page) * kStageRow + cp_blk * 16);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// CBC encryption, staged by the tensor-memory-access engine.  The chains are
// the same (one page per lane).  Lane 0 brings each 8-block chunk of the
// warp's 32 pages in as one 2-D tile, 32 rows of 128 B, with 128-byte
// swizzle: 16-byte piece i of row r lands at piece i ^ (r % 8), so that the
// lanes' 16-byte reads of their own rows fall on distinct banks.  The lanes
// encipher their rows in place, and lane 0 writes the tile back with one
// tensor store, waits until the store has read the buffer, and brings in the
// next chunk.  Neither copy passes through registers or the load/store
// pipe.  Rows past the last page are filled with zeros on the way in and
// clipped on the way out.  Every wait on the tile's mbarrier is bounded; a
// wait that runs out is counted in g_bulk_wait_timeouts, the warp waits once
// more (bounded) for its copy in flight and leaves its remaining pages
// untouched.
// ---------------------------------------------------------------------------
__device__ unsigned int g_bulk_wait_timeouts;

__device__ __forceinline__ bool tile_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t i = 0; i < (1u << 22); i++) {
        uint32_t ok;
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

__device__ __forceinline__ void tile_load(uint32_t sbuf, uint64_t map, int x, int y, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)kTmaWarpBytes)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(sbuf),
        "l"(map), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tile_store(uint64_t map, int x, int y, uint32_t sbuf) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map),
                 "r"(x), "r"(y), "r"(sbuf)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

__device__ __forceinline__ void tile_stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tile_stores_done() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

template <int NR>
__global__ void __launch_bounds__(kCbcEncStagedThreads, 1) cbc_enc_tma_kernel(const __grid_constant__ CbcTmaParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    // kSmemBase + kSmemEnc + warp * 4096: 1024-byte aligned in the shared
    // window, as the 128-byte swizzle wants
    char* buf = smem + kSmemEnc + warp * kTmaWarpBytes;
    const uint32_t sbuf = (uint32_t)__cvta_generic_to_shared(buf);
    const uint32_t bar =
        (uint32_t)__cvta_generic_to_shared(smem + kSmemEnc + kCbcEncStagedMaxWarps * kTmaWarpBytes + warp * 8);
    if (lane == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tensor copies see it initialised
    }
    fill_enc(smem);
    __syncthreads();

    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const ParamKey K{p.rk};
    const uint32_t nchunks = p.bpp / kStageBlocks;
    const uint64_t ngroups = (p.npages + 31) >> 5;
    const uint64_t src_map = reinterpret_cast<uint64_t>(&p.src_map);
    const uint64_t dst_map = reinterpret_cast<uint64_t>(&p.dst_map);
    char* own = buf + lane * 128;  // this lane's row
    uint32_t parity = 0;
    bool ok = true;
    for (uint64_t g = interleaved_warp(); ok && g < ngroups; g += total_warps()) {
        const uint64_t page = (g << 5) + lane;
        uint4 x = page < p.npages ? p.ivs[page] : make_uint4(0, 0, 0, 0);
        const int y = (int)(g << 5);
        if (lane == 0) {
            tile_stores_read();  // the previous group's last store has read the buffer
            tile_load(sbuf, src_map, 0, y, bar);
        }
        for (uint32_t c = 0; c < nchunks; ++c) {
            ok = __all_sync(0xffffffffu, tile_wait(bar, parity));
            if (!ok) break;
            parity ^= 1;
#pragma unroll 1
            for (int i = 0; i < kStageBlocks; i++) {
                uint4* blk = reinterpret_cast<uint4*>(own + ((i ^ (lane & 7)) << 4));
                const uint4 pt = *blk;
                xor4(x, pt.x, pt.y, pt.z, pt.w);
                encrypt_block<NR>(x.x, x.y, x.z, x.w, T, K);
                *blk = x;
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tensor store sees the rows
            __syncwarp();
            if (lane == 0) {
                tile_store(dst_map, (int)(c * 32), y, sbuf);
                if (c + 1 < nchunks) {
                    tile_stores_read();
                    tile_load(sbuf, src_map, (int)((c + 1) * 32), y, bar);
                }
            }
        }
    }
    if (!ok && lane == 0) {
        atomicAdd(&g_bulk_wait_timeouts, 1u);
        tile_wait(bar, parity);  // the load still in flight, bounded
    }
    if (lane == 0) tile_stores_done();
}

// ---------------------------------------------------------------------------
// XTS with ciphertext stealing (IEEE 1619-2007 5.3.2 encryption, 5.4.2
// decryption) for data units of du bytes, du >= 16 and not a multiple of 16:
// m full blocks and a final partial block of b bytes.  One warp per data unit:
// full blocks 0..m-2 go to the lanes (block j with T * alpha^j), then lane 0
// runs the stealing pair, the last full block and the partial block, which
// depend on each other:
//   encryption: CC = enc(P_{m-1}, T a^{m-1});  C_m = CC[0..b);
//               C_{m-1} = enc(P_m || CC[b..16), T a^m)
//   decryption: PP = dec(C_{m-1}, T a^m);  P_m = PP[0..b);
//               P_{m-1} = dec(C_m || PP[b..16), T a^{m-1})
// Unit starts are only as aligned as u * du, so the unit's blocks move through
// 16-, 4- or 1-byte accesses as its start allows.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 load_block(const uint8_t* q, uint32_t align) {
    if (align == 16) return *reinterpret_cast<const uint4*>(q);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        if (align == 4) {
            w[i] = reinterpret_cast<const uint32_t*>(q)[i];
        } else {
            w[i] = (uint32_t)q[4 * i] | (uint32_t)q[4 * i + 1] << 8 | (uint32_t)q[4 * i + 2] << 16 |
                   (uint32_t)q[4 * i + 3] << 24;
        }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void store_block(uint8_t* q, const uint4& v, uint32_t align) {
    if (align == 16) {
        *reinterpret_cast<uint4*>(q) = v;
        return;
    }
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; i++) {
        if (align == 4) {
            reinterpret_cast<uint32_t*>(q)[i] = w[i];
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++) q[4 * i + k] = (uint8_t)(w[i] >> (8 * k));
        }
    }
}

template <int NR, int DIR>
__global__ void __launch_bounds__(kBulkThreads, 1) xts_cts_kernel(const __grid_constant__ CtsParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    if (DIR == 0) fill_enc(smem);
    else fill_dec<true>(smem);
    __syncthreads();

    const uint32_t lane = lane_id();
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const Rep1<2> IS{lane * 4u};
    const Rep1<2> TE{lane * 4u + 128u};
    const ParamKey K{p.rk};
    const ParamKey TK{p.tk};
    const uint64_t m = p.du / 16;
    const uint32_t b = (uint32_t)(p.du % 16);

    auto block = [&](uint4& v, uint32_t t0, uint32_t t1, uint32_t t2, uint32_t t3) {
        xor4(v, t0, t1, t2, t3);
        if (DIR == 0) encrypt_block<NR>(v.x, v.y, v.z, v.w, T, K);
        else decrypt_block<NR>(v.x, v.y, v.z, v.w, T, IS, K);
        xor4(v, t0, t1, t2, t3);
    };

    for (uint64_t u = interleaved_warp(); u < p.units; u += total_warps()) {
        const uint8_t* in = p.src + u * p.du;
        uint8_t* out = p.dst + u * p.du;
        const uint32_t off = (uint32_t)((uintptr_t)in & 15u);
        const uint32_t align = off == 0 ? 16u : (off & 3u) == 0 ? 4u : 1u;
        // E_K2(unit number) on every lane
        const uint64_t unit = p.first_sector + u;
        uint32_t z0 = (uint32_t)unit, z1 = (uint32_t)(unit >> 32), z2 = 0, z3 = 0;
        if (DIR == 0) encrypt_block<NR>(z0, z1, z2, z3, T, TK);
        else encrypt_block<NR>(z0, z1, z2, z3, TE, TK);
        // blocks 0..m-2, lane-strided
        uint32_t t0 = z0, t1 = z1, t2 = z2, t3 = z3;
        gf128_mul_xk(t0, t1, t2, t3, lane);
        for (uint64_t j = lane; j + 1 < m; j += 32) {
            uint4 v = load_block(in + 16 * j, align);
            block(v, t0, t1, t2, t3);
            store_block(out + 16 * j, v, align);
            gf128_mul_x32(t0, t1, t2, t3);
        }
        // the stealing pair: tweaks T a^{m-1} (a*) and T a^m (c*)
        if (lane == 0) {
            uint32_t a0 = z0, a1 = z1, a2 = z2, a3 = z3;
            gf128_mul_xpow(a0, a1, a2, a3, (uint32_t)(m - 1));
            uint32_t c0 = a0, c1 = a1, c2 = a2, c3 = a3;
            gf128_mul_xk(c0, c1, c2, c3, 1);
            uint4 x = load_block(in + 16 * (m - 1), align);
            const uint8_t* tail = in + 16 * m;
            // both inputs are read before anything is written (in-place calls)
            uint32_t yw[4] = {0, 0, 0, 0};
            if (DIR == 0) block(x, a0, a1, a2, a3);  // CC
            else block(x, c0, c1, c2, c3);           // PP
            const uint32_t xw[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int k = 0; k < 16; k++) {
                const uint32_t byte = (uint32_t)k < b ? (uint32_t)tail[k] : (xw[k >> 2] >> (8 * (k & 3))) & 0xffu;
                yw[k >> 2] |= byte << (8 * (k & 3));
            }
            uint4 y = make_uint4(yw[0], yw[1], yw[2], yw[3]);
            if (DIR == 0) block(y, c0, c1, c2, c3);  // C_{m-1}
            else block(y, a0, a1, a2, a3);           // P_{m-1}
            store_block(out + 16 * (m - 1), y, align);
#pragma unroll
            for (int k = 0; k < 16; k++)
                if ((uint32_t)k < b) out[16 * m + k] = (uint8_t)(xw[k >> 2] >> (8 * (k & 3)));
        }
    }
}

template <class P>
using KernelFn = void (*)(P);

// CTAs for a run of 32-block chunks: one per SM, and four chunks each (one per
// SM quarter) before fewer are used.  Filling a CTA's warps first instead left
// most SMs idle in small calls: 1 MiB ran on 64 of them.
inline int grid_for_chunks(uint64_t chunks, int num_sms) {
    const uint64_t ctas = (chunks + 3) / 4;
    return (int)(ctas < (uint64_t)num_sms ? (ctas ? ctas : 1) : num_sms);
}

template <int NR>
KernelFn<BulkParams> pick_bulk(int dir, bool tweak) {
    if (tweak) return dir == 0 ? bulk_kernel<NR, 0, true> : bulk_kernel<NR, 1, true>;
    return dir == 0 ? bulk_kernel<NR, 0, false> : bulk_kernel<NR, 1, false>;
}

KernelFn<BulkParams> bulk_fn(int nr, int dir, bool tweak) {
    switch (nr) {
        case 10: return pick_bulk<10>(dir, tweak);
        case 12: return pick_bulk<12>(dir, tweak);
        case 14: return pick_bulk<14>(dir, tweak);
        default: return nullptr;
    }
}

size_t bulk_smem(int dir, bool tweak) {
    return (dir == 0 ? kSmemEnc : kSmemDec) + (tweak ? kBulkThreads * 16 : 0);
}

KernelFn<CtsParams> cts_fn(int nr, int dir) {
    switch (nr) {
        case 10: return dir ? xts_cts_kernel<10, 1> : xts_cts_kernel<10, 0>;
        case 12: return dir ? xts_cts_kernel<12, 1> : xts_cts_kernel<12, 0>;
        case 14: return dir ? xts_cts_kernel<14, 1> : xts_cts_kernel<14, 0>;
        default: return nullptr;
    }
}

KernelFn<CbcParams> cbc_enc_split_fn(int nr, int lanes) {
    switch (nr) {
        case 10: return lanes == 4 ? cbc_enc_split_kernel<10, 4> : cbc_enc_split_kernel<10, 2>;
        case 12: return lanes == 4 ? cbc_enc_split_kernel<12, 4> : cbc_enc_split_kernel<12, 2>;
        case 14: return lanes == 4 ? cbc_enc_split_kernel<14, 4> : cbc_enc_split_kernel<14, 2>;
        default: return nullptr;
    }
}

KernelFn<CbcParams> cbc_enc_staged_fn(int nr) {
    switch (nr) {
        case 10: return cbc_enc_staged_kernel<10>;
        case 12: return cbc_enc_staged_kernel<12>;
        case 14: return cbc_enc_staged_kernel<14>;
        default: return nullptr;
    }
}

KernelFn<CbcTmaParams> cbc_enc_tma_fn(int nr) {
    switch (nr) {
        case 10: return cbc_enc_tma_kernel<10>;
        case 12: return cbc_enc_tma_kernel<12>;
        case 14: return cbc_enc_tma_kernel<14>;
        default: return nullptr;
    }
}

// cuTensorMapEncodeTiled, found through the runtime (no link against the
// driver library); null if the driver does not provide it.
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return reinterpret_cast<EncodeTiledFn>(f);
    }();
    return fn;
}

// The pages [0, npages) of bpp blocks at base as a 2-D tensor of 32-bit words
// read and written in boxes of 32 words (one 8-block chunk) x 32 pages.
bool page_tile_map(CUtensorMap* m, const void* base, uint64_t npages, uint32_t bpp) {
    EncodeTiledFn enc = encode_tiled();
    if (!enc || npages > 0x7fffffffull) return false;
    const cuuint64_t dim[2] = {(cuuint64_t)bpp * 4, (cuuint64_t)npages};
    const cuuint64_t stride[1] = {(cuuint64_t)bpp * 16};
    const cuuint32_t box[2] = {32, 32};
    const cuuint32_t estride[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void*>(base), dim, stride, box, estride,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

KernelFn<CbcParams> cbc_fn(int nr, bool enc) {
    switch (nr) {
        case 10: return enc ? cbc_enc_kernel<10> : cbc_dec_kernel<10>;
        case 12: return enc ? cbc_enc_kernel<12> : cbc_dec_kernel<12>;
        case 14: return enc ? cbc_enc_kernel<14> : cbc_dec_kernel<14>;
        default: return nullptr;
    }
}

}  // namespace

cudaError_t bulk_wait_timeouts(unsigned int* out) {
    return cudaMemcpyFromSymbol(out, g_bulk_wait_timeouts, sizeof(unsigned int));
}

cudaError_t configure_kernels() {
    for (int nr : {10, 12, 14}) {
        for (int dir = 0; dir < 2; dir++) {
            for (bool tw : {false, true}) {
                cudaError_t e = cudaFuncSetAttribute(bulk_fn(nr, dir, tw), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                     (int)bulk_smem(dir, tw));
                if (e != cudaSuccess) return e;
            }
        }
        cudaError_t e = cudaFuncSetAttribute(cbc_fn(nr, true), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kSmemEnc);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(cbc_fn(nr, false), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemDec);
        if (e != cudaSuccess) return e;
        for (int lanes : {2, 4}) {
            e = cudaFuncSetAttribute(cbc_enc_split_fn(nr, lanes), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemEnc);
            if (e != cudaSuccess) return e;
        }
        e = cudaFuncSetAttribute(cbc_enc_staged_fn(nr), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSmemEncStaged);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(cbc_enc_tma_fn(nr), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemEncTma);
        if (e != cudaSuccess) return e;
        for (int dir = 0; dir < 2; dir++) {
            e = cudaFuncSetAttribute(cts_fn(nr, dir), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)(dir == 0 ? kSmemEnc : kSmemDec));
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

cudaError_t upload_tables(const uint32_t* te0, const uint32_t* td0, const uint32_t* isb4) {
    cudaError_t e = cudaMemcpyToSymbol(g_te0, te0, 1024);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_td0, td0, 1024);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_isb4, isb4, 1024);
    return e;
}

static cudaError_t launch_bulk(const BulkParams& params, int nr, int dir, bool tweak, int num_sms, cudaStream_t s) {
    auto fn = bulk_fn(nr, dir, tweak);
    if (!fn) return cudaErrorInvalidValue;
    BulkParams p = params;
    const uint64_t chunks = (p.nblocks + 31) / 32;
    const int grid = grid_for_chunks(chunks, num_sms);
    if (chunks / grid >= 0xffffffffull) return cudaErrorInvalidValue;
    p.cta_chunks = (uint32_t)(chunks / grid);
    p.cta_rest = (uint32_t)(chunks % grid);
    fn<<<grid, kBulkThreads, bulk_smem(dir, tweak), s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_xts(const BulkParams& p, int nr, int dir, int num_sms, cudaStream_t s) {
    return launch_bulk(p, nr, dir, true, num_sms, s);
}

cudaError_t launch_ecb(const BulkParams& p, int nr, int dir, int num_sms, cudaStream_t s) {
    return launch_bulk(p, nr, dir, false, num_sms, s);
}

cudaError_t launch_cbc_dec(const CbcParams& p, int nr, int num_sms, cudaStream_t s) {
    auto fn = cbc_fn(nr, false);
    if (!fn) return cudaErrorInvalidValue;
    CbcParams q = p;
    const bool in_place = p.src == p.dst;
    const uint64_t items = in_place ? p.npages : (p.npages * p.bpp + 31) / 32;
    const int grid = in_place ? (int)std::min<uint64_t>(items, num_sms) : grid_for_chunks(items, num_sms);
    if (items / grid >= 0xffffffffull) return cudaErrorInvalidValue;
    q.cta_items = (uint32_t)(items / grid);
    q.cta_rest = (uint32_t)(items % grid);
    fn<<<grid, kBulkThreads, kSmemDec, s>>>(q);
    return cudaGetLastError();
}

cudaError_t launch_xts_cts(const CtsParams& p, int nr, int dir, int num_sms, cudaStream_t s) {
    auto fn = cts_fn(nr, dir);
    if (!fn) return cudaErrorInvalidValue;
    const uint64_t warps = kBulkThreads / 32;
    const uint64_t ctas = (p.units + warps - 1) / warps;
    const int grid = (int)(ctas < (uint64_t)num_sms ? (ctas ? ctas : 1) : num_sms);
    fn<<<grid, kBulkThreads, dir == 0 ? kSmemEnc : kSmemDec, s>>>(p);
    return cudaGetLastError();
}

// A group (32 whole-page chains, one warp) is one long serial job, so the
// groups run in waves of warps x SMs, and a last wave that fills only part of
// the warps leaves the SMs' lookup path under-used for a whole chain's time.
// With 16 warps an SM's shared-memory path is kept busy (ncu: 91% of the
// kernel's own lookup bound, the rest being the tail), so a wave of w warps
// per SM costs about max(w, 16) chain-times of lookups.  Pick the warp count
// with the lowest total over the waves (ties: more warps).  1 GiB of 4-KiB
// pages is 8,192 groups: 16 warps take 3.37 waves (the fourth on 37% of the
// warps), 18 take 2.99.  (At 21 warps the register cap drops to 80 and the
// kernel spills.)
int cbc_enc_staged_warps(uint64_t groups, int num_sms) {
    constexpr int kSat = 16;
    const uint64_t sms = (uint64_t)(num_sms > 0 ? num_sms : 1);
    if (groups < kSat * sms) {  // one wave; extra warps only speed the table fill
        const uint64_t w = (groups + sms - 1) / sms;
        return (int)(w < 8 ? 8 : w);
    }
    int best = kCbcEncStagedMaxWarps;
    uint64_t best_cost = UINT64_MAX;
    for (int w = kCbcEncStagedMaxWarps; w >= kSat; --w) {
        const uint64_t per_wave = (uint64_t)w * sms;
        const uint64_t full = groups / per_wave, rest = groups % per_wave;
        const uint64_t last = (rest + sms - 1) / sms;  // warps per SM in the last wave
        const uint64_t cost = full * (uint64_t)w + (rest ? (last > kSat ? last : kSat) : 0);
        if (cost < best_cost) {
            best_cost = cost;
            best = w;
        }
    }
    return best;
}

// The last pair of tensor maps made, for calls that repeat on the same buffers
// (encoding one costs microseconds of host time).
struct TileMapCache {
    std::mutex mu;
    bool valid = false;
    const void* src = nullptr;
    const void* dst = nullptr;
    uint64_t npages = 0;
    uint32_t bpp = 0;
    CUtensorMap src_map, dst_map;
};

bool page_tile_maps(CbcTmaParams* t, const CbcParams& p) {
    static TileMapCache c;
    std::lock_guard<std::mutex> lk(c.mu);
    if (!(c.valid && c.src == p.src && c.dst == p.dst && c.npages == p.npages && c.bpp == p.bpp)) {
        c.valid = page_tile_map(&c.src_map, p.src, p.npages, p.bpp) && page_tile_map(&c.dst_map, p.dst, p.npages, p.bpp);
        if (!c.valid) return false;
        c.src = p.src;
        c.dst = p.dst;
        c.npages = p.npages;
        c.bpp = p.bpp;
    }
    t->src_map = c.src_map;
    t->dst_map = c.dst_map;
    return true;
}

cudaError_t launch_cbc_enc(const CbcParams& p, int nr, int num_sms, cudaStream_t s) {
    // Few pages are a chain's latency, which two or four lanes per page
    // shorten; many are the lookups' rate, which one lane per page uses best.
    // 4-KiB pages, AES-128, one / two / four lanes: 8 pages per SM 145 / 107 /
    // 103 us, 32 pages 145 / 109 / 107, 64 pages 147 / 121 / 121, 128 pages 153
    // / 152 / 180, 160 pages 206 / 182 / 288, 192 pages 208 / 207 / 295, 224
    // pages 215 / 248 / 316.  Pages that cannot be staged cross later (4112 B,
    // AES-256: 224 pages 299 / 286, 256 pages 306 / 309).
    const uint64_t sms = (uint64_t)(num_sms > 0 ? num_sms : 1);
    const int lanes = p.npages <= 32 * sms ? 4 : p.npages <= (p.bpp % kStageBlocks ? 240 : 192) * sms ? 2 : 1;
    if (lanes > 1) {
        auto fn = cbc_enc_split_fn(nr, lanes);
        if (!fn) return cudaErrorInvalidValue;
        const uint64_t teams = (p.npages + 32 / lanes - 1) / (32 / lanes);
        fn<<<(int)std::min<uint64_t>(teams, sms), kCbcSplitThreads, kSmemEnc, s>>>(p);
        return cudaGetLastError();
    }
    // The tensor tiles take a seventh of the staging traffic off the
    // shared-memory path, which pays once that path is the bound: from 12
    // groups of 32 pages per SM (measured at 4-KiB pages: 8 groups per SM
    // 227 us staged through registers against 232 us in tiles, 16 groups
    // 389 against 355 us).  Below that a launch is a chain's latency either
    // way, and the tiles' two tensor maps would only add host time.
    const uint64_t groups = (p.npages + 31) / 32;
    if (p.bpp % kStageBlocks == 0 && groups >= 12 * sms) {
        CbcTmaParams t;
        std::memset(&t, 0, sizeof(t));
        auto fn = cbc_enc_tma_fn(nr);
        if (fn && page_tile_maps(&t, p)) {
            t.ivs = p.ivs;
            t.npages = p.npages;
            t.bpp = p.bpp;
            std::memcpy(t.rk, p.rk, sizeof(t.rk));
            const int grid = num_sms;
            const int warps = cbc_enc_staged_warps(groups, num_sms);
            fn<<<grid, warps * 32, kSmemEncTma, s>>>(t);
            return cudaGetLastError();
        }
    }
    if (p.bpp % kStageBlocks == 0) {
        auto fn = cbc_enc_staged_fn(nr);
        if (!fn) return cudaErrorInvalidValue;
        const int grid = (int)(groups < (uint64_t)num_sms ? (groups ? groups : 1) : num_sms);
        const int warps = cbc_enc_staged_warps(groups, num_sms);
        fn<<<grid, warps * 32, kSmemEnc + warps * kStageWarpSmem, s>>>(p);
        return cudaGetLastError();
    }
    auto fn = cbc_fn(nr, true);
    if (!fn) return cudaErrorInvalidValue;
    // a 32-page group is a heavy work item (32 chains of whole pages): give
    // every SM work as soon as there are as many groups as SMs
    const int grid = (int)(groups < (uint64_t)num_sms ? (groups ? groups : 1) : num_sms);
    fn<<<grid, kBulkThreads, kSmemEnc, s>>>(p);
    return cudaGetLastError();
}

}  // namespace kgpu
