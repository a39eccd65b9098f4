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
#include <atomic>
#include <cstring>
#include <type_traits>
#include <mutex>

#include "aes_device.cuh"
#include "bitslice_device.cuh"
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

// Programmatic dependent launch.  A launch's tables do not depend on the work
// queued before it, so the kernels are launched with programmatic stream
// serialisation: next_may_start() lets the next such launch of the stream put
// its CTAs on SMs that have room and fill their tables while this one runs,
// and wait_for_previous() holds every CTA, before it touches a caller's buffer,
// until all earlier work of the stream has completed and its writes are
// visible.  Every CTA waits, so a launch never completes before the one it
// follows.  GPU time of back-to-back calls without and with it: 4 KiB of
// AES-256-XTS 7.2 / 4.4 us, 1 MiB 8.2 / 5.5, 16 MiB 30.8 / 28.4, 64 MiB of
// AES-128-CBC decryption 81.9 / 77.5.  A waiting CTA keeps its SM from other
// streams, so CBC encryption, whose chains take 100 us and more, lets the next
// launch start only when its first warps are at their end (10,000 mixed requests
// of 4 KiB to 8 MiB, one launch each on eight streams: 96 -> 163 GB/s).
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

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
template <int NR, int DIR, bool TWEAK, int WARPS>
__device__ __forceinline__ void bulk_chunks(const BulkParams& p, uint4* tweaks, uint64_t first, uint32_t own) {
    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    constexpr uint32_t kWarps = WARPS;
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const Rep1<2> IS{lane * 4u};
    const Rep1<2> TE{lane * 4u + 128u};
    const ParamKey K{p.rk};
    const ParamKey TK{p.tk};

    // this warp's part of the run
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
    const uint32_t gthreads = shared ? kWarps * 32u : 32u;
    const uint32_t gwarp = shared ? warp : 0u, gwarps = shared ? kWarps : 1u;
    uint4* tw = tweaks + (shared ? 0u : warp * 32u);
    auto group_sync = [&]() {
        if (!shared) __syncwarp();
        else if (WARPS * 32 == kBulkThreads) __syncthreads();
        else asm volatile("bar.sync 1, %0;" ::"n"(WARPS * 32) : "memory");  // the mixed kernel's table warps
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

// This CTA's run of 32-block chunks.
__device__ __forceinline__ uint64_t cta_first(const BulkParams& p) {
    return (uint64_t)p.cta_chunks * blockIdx.x + min(blockIdx.x, p.cta_rest);
}
__device__ __forceinline__ uint32_t cta_own(const BulkParams& p) {
    return p.cta_chunks + (blockIdx.x < p.cta_rest ? 1u : 0u);
}

template <int NR, int DIR, bool TWEAK>
__global__ void __launch_bounds__(kBulkThreads, 1) bulk_kernel(const __grid_constant__ BulkParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;  // uniform over the CTA; refused at init
    next_may_start();
    if (DIR == 0) fill_enc(smem);
    else fill_dec<TWEAK>(smem);
    wait_for_previous();
    __syncthreads();
    uint4* tweaks = reinterpret_cast<uint4*>(smem + (DIR == 0 ? kSmemEnc : kSmemDec));
    bulk_chunks<NR, DIR, TWEAK, kBulkThreads / 32>(p, tweaks, cta_first(p), cta_own(p));
}

// ---------------------------------------------------------------------------
// Large XTS and ECB calls on two pipes at once.  The lookups keep the
// shared-memory path 97% busy and leave two thirds of the ALU pipe and a third
// of the issue slots idle, so four warps of every CTA encipher part of its run
// without lookups, bitsliced: 32 blocks per lane as 128 bit-planes (see
// bitslice_device.cuh).  Their round keys are masks in the parameter bank and
// their spills are outside the rounds, so that they stay off the shared-memory
// path; a warp beside its SM quarter's four table warps takes about 140 us for
// a span of 1,024 blocks with AES-256, 43 with the quarter to itself.  The 16
// table warps (as fast as 32 here) take the rest of the run as bulk_kernel
// does.  The split is fixed by the launch (mix_spans): the spans come from the
// start of the run, where all blocks exist.
//
// The rounds of both parts are as they measured best.  Table rounds as a loop,
// to leave the instruction cache to the planes, wait for their keys (1 GiB of
// AES-256: 1,660 us with a tenth on planes, 1,496 unrolled); with 8 or 12 table
// warps of two blocks a lane the planes go faster, but the tables lose more
// (1,637 / 1,508 us); plane masks in shared memory cost 11 us of 1,489.
// Tables alone / mixed: AES-256-XTS of 1 GiB 1,584 / 1,474 us, 300 MiB 471 / 439,
// 112 MiB 181 / 172; AES-128-XTS of 1 GiB 1,155 / 1,098; ECB of 1 GiB 1,573 /
// 1,427 and 1,146 / 1,046.  Decryption, whose inverse S-box and InvMixColumns are
// a fifth more work on the planes: AES-256-XTS of 1 GiB 1,591 / 1,524, 130 MiB
// 208 / 201; AES-128-XTS 1,165 / 1,130; ECB 1,582 / 1,471 and 1,156 / 1,071.
// ---------------------------------------------------------------------------

__device__ __forceinline__ void load_span(uint32_t (&S)[128], const uint4* in) {
#pragma unroll
    for (int i = 0; i < 32; i++) {
        const uint4 v = in[32 * i];
        S[i] = v.x;
        S[32 + i] = v.y;
        S[64 + i] = v.z;
        S[96 + i] = v.w;
    }
}

template <int NR, int DIR>
__device__ __forceinline__ void cipher_span(uint32_t (&S)[128], const uint32_t* masks) {
#pragma unroll
    for (int q = 0; q < 4; q++) transpose32(S + 32 * q);
    if constexpr (DIR == 0) bs_encrypt<NR, false>(S, masks);
    else bs_decrypt<NR>(S, masks);
#pragma unroll
    for (int q = 0; q < 4; q++) transpose32(S + 32 * q);
}

// Blocks [b0, b0 + 1024), bitsliced; lane l holds blocks l, l + 32, ... .  tw:
// 32 words of shared memory for the E_K2 of the span's data units, which has
// at most 32 as a unit is at least 32 blocks and b0 a multiple of 32.
template <int NR, int DIR, bool TWEAK>
__device__ __forceinline__ void bitsliced_span(const MixParams& mp, uint4* tw, uint64_t b0) {
    const BulkParams& p = mp.b;
    const uint32_t lane = lane_id();
    const uint32_t bps = p.bps;
    uint32_t u0 = 0, j0 = 0;
    uint4 t0 = make_uint4(0, 0, 0, 0);
    if constexpr (TWEAK) {
        const uint64_t unit0 = div_small(b0, bps);
        const uint32_t q = (uint32_t)(b0 - unit0 * bps) + lane;
        const uint64_t unit = p.first_sector + unit0 + lane;
        uint4 z = make_uint4((uint32_t)unit, (uint32_t)(unit >> 32), 0, 0);
        if constexpr (DIR == 0)
            encrypt_block<NR>(z.x, z.y, z.z, z.w, Rep4{lane * 4u, lane * 4u + 128u}, ParamKey{p.tk});
        else
            encrypt_block<NR>(z.x, z.y, z.z, z.w, Rep1<2>{lane * 4u + 128u}, ParamKey{p.tk});
        __syncwarp();  // the last span's have been read
        tw[lane] = z;
        __syncwarp();
        u0 = q / bps;
        j0 = q - u0 * bps;
        t0 = tw[u0];
        gf128_mul_xpow(t0.x, t0.y, t0.z, t0.w, j0);
    }
    uint32_t S[128];
    load_span(S, p.src + b0 + lane);
    auto whiten = [&]() {
        uint32_t u = u0, j = j0;
        uint4 t = t0;
#pragma unroll
        for (int i = 0; i < 32; i++) {
            S[i] ^= t.x;
            S[32 + i] ^= t.y;
            S[64 + i] ^= t.z;
            S[96 + i] ^= t.w;
            if (i == 31) break;
            j += 32;
            if (j >= bps) {
                j -= bps;
                t = tw[++u];
                gf128_mul_xk(t.x, t.y, t.z, t.w, j);
            } else {
                gf128_mul_x32(t.x, t.y, t.z, t.w);
            }
        }
    };
    if constexpr (TWEAK) whiten();
    cipher_span<NR, DIR>(S, mp.masks);
    if constexpr (TWEAK) whiten();
    uint4* out = p.dst + b0 + lane;
#pragma unroll
    for (int i = 0; i < 32; i++) out[32 * i] = make_uint4(S[i], S[32 + i], S[64 + i], S[96 + i]);
}

template <int NR, int DIR, bool TWEAK>
__global__ void __launch_bounds__(kMixThreads, 1) mixed_kernel(const __grid_constant__ MixParams mp) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    next_may_start();
    if (DIR == 0) fill_enc(smem);
    else fill_dec<TWEAK>(smem);
    wait_for_previous();
    __syncthreads();
    uint4* tweaks = reinterpret_cast<uint4*>(smem + (DIR == 0 ? kSmemEnc : kSmemDec));
    const uint64_t first = cta_first(mp.b);
    const uint32_t spans = mp.spans * kMixPlaneWarps;
    const uint32_t warp = threadIdx.x >> 5;
    if (warp < kMixTableWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kMixTableRegs));
        bulk_chunks<NR, DIR, TWEAK, kMixTableWarps>(mp.b, tweaks, first + kMixSpanChunks * spans,
                                                    cta_own(mp.b) - kMixSpanChunks * spans);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kMixPlaneRegs));
#pragma unroll 1
        for (uint32_t s = warp - kMixTableWarps; s < spans; s += kMixPlaneWarps)
            bitsliced_span<NR, DIR, TWEAK>(mp, tweaks + warp * 32u, (first + (uint64_t)kMixSpanChunks * s) << 5);
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
template <int NR, int WARPS>
__device__ __forceinline__ void cbc_dec_chunks(const CbcParams& p, uint64_t b0, uint64_t bend) {
    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    constexpr uint32_t kWarps = WARPS;
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const Rep1<2> IS{lane * 4u};
    const ParamKey K{p.rk};

    const uint32_t bpp = p.bpp;
    const uint32_t chunks = (uint32_t)((bend - b0 + 31) >> 5);
    const uint32_t a = (uint32_t)((uint64_t)chunks * warp / kWarps);
    const uint32_t e = (uint32_t)((uint64_t)chunks * (warp + 1) / kWarps);
    uint64_t blk = b0 + ((uint64_t)a << 5) + lane;
    uint64_t page = div_small(blk, bpp);
    uint32_t j = (uint32_t)(blk - page * bpp);
    const bool some = a < e && blk < bend;
    uint4 carry = some && lane == 0 && j ? p.src[blk - 1] : make_uint4(0, 0, 0, 0);
    uint4 nxt = some ? p.src[blk] : make_uint4(0, 0, 0, 0);
    if (WARPS * 32 == kBulkThreads) __syncthreads();  // the tables are filled and every carry is read

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

// This CTA's blocks [b0, bend): pages in place, else 32-block chunks.
__device__ __forceinline__ void cta_blocks(const CbcParams& p, uint64_t& b0, uint64_t& bend) {
    const uint64_t item = p.src == p.dst ? p.bpp : 32u;
    const uint64_t first = (uint64_t)p.cta_items * blockIdx.x + min(blockIdx.x, p.cta_rest);
    const uint32_t own = p.cta_items + (blockIdx.x < p.cta_rest ? 1u : 0u);
    b0 = first * item;
    bend = min(b0 + own * item, p.npages * p.bpp);
}

template <int NR>
__global__ void __launch_bounds__(kBulkThreads, 1) cbc_dec_kernel(const __grid_constant__ CbcParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    next_may_start();
    fill_dec<false>(smem);
    wait_for_previous();
    uint64_t b0, bend;
    cta_blocks(p, b0, bend);
    cbc_dec_chunks<NR, kBulkThreads / 32>(p, b0, bend);
}

// Large CBC decryption out of place on tables and bit-planes, as mixed_kernel.
// A span's lanes read the block before each of theirs again once they have
// deciphered it; pages are of at least 32 blocks, so that a lane enters at most
// one from one block to its next.  4-KiB pages, tables alone / mixed: AES-128 of
// 1 GiB 1,189 / 1,121 us, of 130 MiB 156 / 150; AES-256 1,616 / 1,541.
template <int NR>
__global__ void __launch_bounds__(kMixThreads, 1) mixed_cbc_dec_kernel(const __grid_constant__ MixCbcParams mp) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    next_may_start();
    fill_dec<false>(smem);
    wait_for_previous();
    __syncthreads();
    const CbcParams& p = mp.c;
    uint64_t b0, bend;
    cta_blocks(p, b0, bend);
    const uint32_t spans = mp.spans * kMixPlaneWarps;
    const uint32_t warp = threadIdx.x >> 5;
    if (warp < kMixTableWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kMixTableRegs));
        cbc_dec_chunks<NR, kMixTableWarps>(p, b0 + (uint64_t)kBsSpan * spans, bend);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kMixPlaneRegs));
        const uint32_t bpp = p.bpp;
#pragma unroll 1
        for (uint32_t s = warp - kMixTableWarps; s < spans; s += kMixPlaneWarps) {
            const uint64_t n = b0 + (uint64_t)kBsSpan * s + lane_id();
            uint32_t S[128];
            load_span(S, p.src + n);
            cipher_span<NR, 1>(S, mp.masks);
            uint64_t page = div_small(n, bpp);
            uint32_t j = (uint32_t)(n - page * bpp);
#pragma unroll
            for (int i = 0; i < 32; i++) {
                const uint4 prev = j ? p.src[n + 32 * i - 1] : p.ivs[page];
                p.dst[n + 32 * i] =
                    make_uint4(S[i] ^ prev.x, S[32 + i] ^ prev.y, S[64 + i] ^ prev.z, S[96 + i] ^ prev.w);
                j += 32;
                if (j >= bpp) {
                    j -= bpp;
                    page++;
                }
            }
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
    wait_for_previous();
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
    if (threadIdx.x < 32) next_may_start();
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
    wait_for_previous();
    constexpr int kCols = 4 / LANES;              // columns per lane
    constexpr uint32_t kPages = 32 / LANES;       // pages per warp
    using Piece = std::conditional_t<kCols == 1, uint32_t, uint2>;
    const uint32_t lane = lane_id();
    const uint32_t c = lane & (LANES - 1u), team = lane & ~(LANES - 1u);
    const Rep4Permute T{lane * 4u, lane * 4u + 128u};
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
        const uint32_t late = threadIdx.x < 32 && g + total_warps() >= ngroups ? max(bpp, 8u) - 8u : bpp;
        for (uint32_t i = 0; i < bpp; ++i) {
            if (i == late) next_may_start();
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
//
// PERMUTE: calls over the host link whose time is a chain's latency build their
// addresses by byte permutes, which take less of it (64 pages of 64 KiB, AES-128:
// 2,386 us by dp2a, 2,306 this way).
// ---------------------------------------------------------------------------
constexpr int kStageBlocks = 8;
static_assert(kStageBlocks == kLineBlocks, "a staged chunk is a 128-byte line");
constexpr int kStageRow = kStageBlocks * 16 + 16;  // one page's 8 blocks, padded against bank conflicts
constexpr int kStageWarpBytes = 32 * kStageRow;
static_assert(kStageWarpBytes == kStageWarpSmem, "staging area size");

template <int NR, bool PERMUTE>
__global__ void __launch_bounds__(kCbcEncStagedThreads, 1) cbc_enc_staged_kernel(const __grid_constant__ CbcParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    fill_enc(smem);
    wait_for_previous();
    __syncthreads();

    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    const Rep4Tables<PERMUTE> T{lane * 4u, lane * 4u + 128u};
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
    if (warp == 0) next_may_start();
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
    wait_for_previous();
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
    if (warp == 0) next_may_start();
    if (!ok && lane == 0) {
        atomicAdd(&g_bulk_wait_timeouts, 1u);
        tile_wait(bar, parity);  // the load still in flight, bounded
    }
    if (lane == 0) tile_stores_done();
}

// ---------------------------------------------------------------------------
// XTS with ciphertext stealing (IEEE 1619-2007 5.3.2 encryption, 5.4.2
// decryption) for data units of du bytes, du >= 16 and not a multiple of 16:
// m full blocks and a final partial block of b bytes.  The last full block and
// the partial block depend on each other:
//   encryption: CC = enc(P_{m-1}, T a^{m-1});  C_m = CC[0..b);
//               C_{m-1} = enc(P_m || CC[b..16), T a^m)
//   decryption: PP = dec(C_{m-1}, T a^m);  P_m = PP[0..b);
//               P_{m-1} = dec(C_m || PP[b..16), T a^{m-1})
// A CTA owns a run of units and takes them in phases of one unit per thread:
// the threads encipher the units' tweaks, then the m full blocks of all units
// as one sequence of 32-block chunks split over the warps (the CC or PP of
// each unit stays in shared memory), then the second block of the pair, one
// unit per thread.  So every lane has a block in each of the three passes and
// the lookups are the bound; with one warp per unit, two of the warp's 34
// enciphering steps on a 520-byte unit worked for one lane only, one more for
// the tweak, and a 100-byte unit filled 6 of 32 lanes.
// 32,768 units of 520 B, AES-256: 120.4 -> 34.9 us (488.9 GB/s); 8,192 of 527 B,
// decryption: 41.1 -> 18.5 us; 10,485 of 100 B, AES-128: 32.8 -> 8.2 us.
//
// Unit starts are only as aligned as u * du.  Units of a multiple of 8 bytes
// move in 8-byte accesses; others are read as the two aligned 16-byte words
// that hold a block and shifted into place, and written as aligned 4-byte words
// with smaller pieces at their ends.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint4 load_tail_word(const uint8_t* q, const uint8_t* end) {
    // the aligned word at q, of which only the bytes before end are there
    uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < 16; k++)
        if (q + k < end) w[k >> 2] |= (uint32_t)q[k] << (8 * (k & 3));
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// The 16 bytes at q as loaded (lo, hi), and put in place by settle().
struct RawBlock {
    uint4 lo, hi;
};

__device__ __forceinline__ RawBlock load_raw(const uint8_t* q, const uint8_t* end, bool by8) {
    RawBlock r;
    r.hi = make_uint4(0, 0, 0, 0);
    if (by8) {
        const uint2 x = *reinterpret_cast<const uint2*>(q);
        const uint2 y = q + 16 <= end ? *reinterpret_cast<const uint2*>(q + 8) : make_uint2(0, 0);
        r.lo = make_uint4(x.x, x.y, y.x, y.y);
        return r;
    }
    const uint32_t off = (uint32_t)((uintptr_t)q & 15u);
    const uint8_t* a = q - off;
    r.lo = a + 16 <= end ? *reinterpret_cast<const uint4*>(a) : load_tail_word(a, end);
    if (off && a + 16 < end) r.hi = a + 32 <= end ? *reinterpret_cast<const uint4*>(a + 16) : load_tail_word(a + 16, end);
    return r;
}

__device__ __forceinline__ uint4 settle(const RawBlock& r, const uint8_t* q, bool by8) {
    if (by8) return r.lo;
    const uint32_t off = (uint32_t)((uintptr_t)q & 15u), sh = (off & 3u) * 8u;
    const bool s1 = (off & 4u) != 0, s2 = (off & 8u) != 0;
    uint32_t w[8] = {r.lo.x, r.lo.y, r.lo.z, r.lo.w, r.hi.x, r.hi.y, r.hi.z, r.hi.w};
#pragma unroll
    for (int i = 0; i < 6; i++) w[i] = s2 ? w[i + 2] : w[i];
#pragma unroll
    for (int i = 0; i < 5; i++) w[i] = s1 ? w[i + 1] : w[i];
    return make_uint4(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh),
                      __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh));
}

__device__ __forceinline__ void store_any(uint8_t* q, const uint4& v, bool by8) {
    if (by8) {
        reinterpret_cast<uint2*>(q)[0] = make_uint2(v.x, v.y);
        reinterpret_cast<uint2*>(q)[1] = make_uint2(v.z, v.w);
        return;
    }
    const uint32_t k = (uint32_t)((uintptr_t)q & 3u);
    if (k == 0) {
        uint32_t* o = reinterpret_cast<uint32_t*>(q);
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
        return;
    }
    const uint32_t h = 4 - k;  // bytes up to the first aligned word
    if (h & 1u) {
        q[0] = (uint8_t)v.x;
        if (h == 3) *reinterpret_cast<uint16_t*>(q + 1) = (uint16_t)(v.x >> 8);
    } else {
        *reinterpret_cast<uint16_t*>(q) = (uint16_t)v.x;
    }
    uint32_t* o = reinterpret_cast<uint32_t*>(q + h);
    o[0] = __funnelshift_r(v.x, v.y, 8 * h);
    o[1] = __funnelshift_r(v.y, v.z, 8 * h);
    o[2] = __funnelshift_r(v.z, v.w, 8 * h);
    const uint32_t rest = v.w >> (8 * h);  // the last k bytes
    uint8_t* t = q + 16 - k;
    if (k & 2u) {
        *reinterpret_cast<uint16_t*>(t) = (uint16_t)rest;
        if (k == 3) t[2] = (uint8_t)(rest >> 16);
    } else {
        t[0] = (uint8_t)rest;
    }
}

// The first b (< 16) bytes of v.
__device__ __forceinline__ void store_part(uint8_t* q, const uint4& v, uint32_t b) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const bool by4 = ((uintptr_t)q & 3u) == 0;
#pragma unroll
    for (uint32_t i = 0; i < 4; i++) {
        if (by4 && b >= 4 * i + 4) {
            reinterpret_cast<uint32_t*>(q)[i] = w[i];
        } else {
#pragma unroll
            for (uint32_t k = 0; k < 4; k++)
                if (4 * i + k < b) q[4 * i + k] = (uint8_t)(w[i] >> (8 * k));
        }
    }
}

// Bytes [0, b) of x and [b, 16) of y.
__device__ __forceinline__ uint4 splice(const uint4& x, const uint4& y, uint32_t b) {
    auto word = [&](uint32_t xw, uint32_t yw, uint32_t i) {
        const uint32_t mask = b >= 4 * i + 4 ? ~0u : b <= 4 * i ? 0u : (1u << (8 * (b - 4 * i))) - 1u;
        return (xw & mask) | (yw & ~mask);
    };
    return make_uint4(word(x.x, y.x, 0), word(x.y, y.y, 1), word(x.z, y.z, 2), word(x.w, y.w, 3));
}

template <int NR, int DIR>
__global__ void __launch_bounds__(kCtsThreads, 1) xts_cts_kernel(const __grid_constant__ CtsParams p) {
    extern __shared__ __align__(128) char smem[];
    if (!smem_layout_ok(smem)) return;
    next_may_start();
    if (DIR == 0) fill_enc(smem);
    else fill_dec<true>(smem);
    wait_for_previous();
    __syncthreads();

    const uint32_t lane = lane_id();
    const uint32_t warp = threadIdx.x >> 5;
    constexpr uint32_t kWarps = kCtsThreads / 32;
    const Rep4 T{lane * 4u, lane * 4u + 128u};
    const Rep1<2> IS{lane * 4u};
    const Rep1<2> TE{lane * 4u + 128u};
    const ParamKey K{p.rk};
    const ParamKey TK{p.tk};
    uint4* tw = reinterpret_cast<uint4*>(smem + (DIR == 0 ? kSmemEnc : kSmemDec));  // E_K2 of the phase's units
    uint4* cc = tw + kCtsThreads;                                                   // CC / PP of its units

    const uint64_t du = p.du;
    const uint32_t m = (uint32_t)(du / 16), b = (uint32_t)(du % 16);
    const bool by8 = b == 8;
    const uint8_t* end = p.src + p.units * du;
    const uint64_t first = (uint64_t)p.cta_units * blockIdx.x + min((uint64_t)blockIdx.x, (uint64_t)p.cta_rest);
    const uint64_t own = p.cta_units + (blockIdx.x < p.cta_rest ? 1u : 0u);
    const uint32_t most = max(1u, min((uint32_t)kCtsThreads, (1u << 30) / m));  // units per phase

    auto cipher = [&](uint4& v, const uint4& t) {
        xor4(v, t.x, t.y, t.z, t.w);
        if (DIR == 0) encrypt_block<NR>(v.x, v.y, v.z, v.w, T, K);
        else decrypt_block<NR>(v.x, v.y, v.z, v.w, T, IS, K);
        xor4(v, t.x, t.y, t.z, t.w);
    };

    for (uint64_t done = 0; done < own;) {
        const uint32_t n = (uint32_t)min(own - done, (uint64_t)most);
        const uint64_t unit0 = first + done;
        if (done) __syncthreads();  // the last phase's tw and cc have been read
        if (warp * 32 < n) {
            const uint64_t unit = p.first_sector + unit0 + threadIdx.x;
            uint4 z = make_uint4((uint32_t)unit, (uint32_t)(unit >> 32), 0, 0);
            if (DIR == 0) encrypt_block<NR>(z.x, z.y, z.z, z.w, T, TK);
            else encrypt_block<NR>(z.x, z.y, z.z, z.w, TE, TK);
            tw[threadIdx.x] = z;
        }
        __syncthreads();

        // the full blocks: block j of unit u is item u * m + j
        const uint64_t items = (uint64_t)n * m;
        const uint32_t chunks = (uint32_t)((items + 31) >> 5);
        const uint32_t a = (uint32_t)((uint64_t)chunks * warp / kWarps);
        const uint32_t e = (uint32_t)((uint64_t)chunks * (warp + 1) / kWarps);
        if (a < e) {
            uint64_t q = ((uint64_t)a << 5) + lane;
            const bool some = q < items;
            uint32_t u = some ? (uint32_t)div_small(q, m) : 0u;
            uint32_t j = some ? (uint32_t)(q - (uint64_t)u * m) : 0u;
            uint64_t off = (unit0 + u) * du + 16ull * j;
            uint4 t = tw[u];
            gf128_mul_xpow(t.x, t.y, t.z, t.w, j);
            RawBlock nxt{};
            if (some) nxt = load_raw(p.src + off, end, by8);
            for (uint32_t i = a; i < e; ++i) {
                uint4 v = settle(nxt, p.src + off, by8);
                const bool valid = q < items;
                // where this lane goes next; its block is fetched meanwhile
                uint32_t un = u, jn = j + 32;
                uint64_t offn = off + 512;
                q += 32;
                const bool more = i + 1 < e && q < items;
                const bool crossed = jn >= m;
                if (more && crossed) {
                    const uint32_t ns = m >= 32 ? 1u : jn / m;
                    un += ns;
                    jn -= ns * m;
                    offn = (unit0 + un) * du + 16ull * jn;
                }
                if (more) nxt = load_raw(p.src + offn, end, by8);
                const bool last = j + 1 == m;
                uint4 tv = t;
                if (DIR == 1 && last) gf128_mul_xk(tv.x, tv.y, tv.z, tv.w, 1);
                cipher(v, tv);
                if (valid) {
                    if (last) cc[u] = v;
                    else store_any(p.dst + off, v, by8);
                }
                if (more) {
                    if (crossed) {
                        t = tw[un];
                        gf128_mul_xk(t.x, t.y, t.z, t.w, jn);
                    } else {
                        gf128_mul_x32(t.x, t.y, t.z, t.w);
                    }
                }
                u = un;
                j = jn;
                off = offn;
            }
        }
        __syncthreads();

        // the pair's second block, one unit per thread
        if (warp * 32 < n) {
            const bool valid = threadIdx.x < n;
            const uint32_t u = valid ? threadIdx.x : 0u;
            const uint64_t off = (unit0 + u) * du + 16ull * (m - 1);
            uint4 t = tw[u];
            gf128_mul_xpow(t.x, t.y, t.z, t.w, DIR == 0 ? m : m - 1);
            const uint4 x = cc[u];
            const uint8_t* tail = p.src + off + 16;
            uint4 y = splice(settle(load_raw(tail, end, by8), tail, by8), x, b);
            cipher(y, t);
            if (valid) {
                store_part(p.dst + off + 16, x, b);
                store_any(p.dst + off, y, by8);
            }
        }
        done += n;
    }
}

template <class P>
using KernelFn = void (*)(P);

// Launch with programmatic stream serialisation (see next_may_start).
template <class P>
cudaError_t launch(KernelFn<P> fn, int grid, int threads, size_t smem, cudaStream_t s, const P& p) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, p);
}

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

template <int NR>
KernelFn<MixParams> pick_mixed(int dir, bool tweak) {
    if (tweak) return dir == 0 ? mixed_kernel<NR, 0, true> : mixed_kernel<NR, 1, true>;
    return dir == 0 ? mixed_kernel<NR, 0, false> : mixed_kernel<NR, 1, false>;
}

KernelFn<MixParams> mixed_fn(int nr, int dir, bool tweak) {
    switch (nr) {
        case 10: return pick_mixed<10>(dir, tweak);
        case 12:  // there is no XTS-AES-192
            if (tweak) return nullptr;
            return dir == 0 ? mixed_kernel<12, 0, false> : mixed_kernel<12, 1, false>;
        case 14: return pick_mixed<14>(dir, tweak);
        default: return nullptr;
    }
}

KernelFn<MixCbcParams> mixed_cbc_dec_fn(int nr) {
    switch (nr) {
        case 10: return mixed_cbc_dec_kernel<10>;
        case 12: return mixed_cbc_dec_kernel<12>;
        case 14: return mixed_cbc_dec_kernel<14>;
        default: return nullptr;
    }
}

size_t mixed_smem(int dir) { return (dir == 0 ? kSmemEnc : kSmemDec) + kMixTweakBytes; }

// The mixed kernels that may be launched, one bit each: those compiled to the
// register count that the register shares of their warps are drawn from (a
// share beyond it would wait for ever).  Another compiler may give another
// count; calls then stay on the table kernels, which take every size.
std::atomic<uint32_t> g_mixed_usable{0};

constexpr uint32_t mixed_bit(int nr, int dir, bool tweak) { return 1u << ((nr - 10) * 2 + dir * 2 + (tweak ? 1 : 0)); }
constexpr uint32_t mixed_cbc_dec_bit(int nr) { return 1u << (12 + (nr - 10) / 2); }

template <class P>
cudaError_t configure_mixed(KernelFn<P> fn, size_t smem, uint32_t bit) {
    if (!fn) return cudaSuccess;
    cudaFuncAttributes attr;
    cudaError_t e = cudaFuncGetAttributes(&attr, fn);
    if (e != cudaSuccess) return e;
    if (attr.numRegs != kMixLaunchRegs) {
        g_mixed_usable.fetch_and(~bit);
        return cudaSuccess;
    }
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) g_mixed_usable.fetch_or(bit);
    return e;
}

void plane_masks(uint32_t* masks, const uint32_t* rk, int nr) {
    for (int i = 0; i < 128 * (nr + 1); i++) masks[i] = (rk[i >> 5] >> (i & 31)) & 1u ? ~0u : 0u;
}

size_t cts_smem(int dir) { return (dir == 0 ? kSmemEnc : kSmemDec) + kCtsThreads * 32; }

KernelFn<CtsParams> cts_fn(int nr, int dir) {
    switch (nr) {
        case 10: return dir ? xts_cts_kernel<10, 1> : xts_cts_kernel<10, 0>;
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

KernelFn<CbcParams> cbc_enc_staged_fn(int nr, bool permute) {
    switch (nr) {
        case 10: return permute ? cbc_enc_staged_kernel<10, true> : cbc_enc_staged_kernel<10, false>;
        case 12: return permute ? cbc_enc_staged_kernel<12, true> : cbc_enc_staged_kernel<12, false>;
        case 14: return permute ? cbc_enc_staged_kernel<14, true> : cbc_enc_staged_kernel<14, false>;
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
                e = configure_mixed(mixed_fn(nr, dir, tw), mixed_smem(dir), mixed_bit(nr, dir, tw));
                if (e != cudaSuccess) return e;
            }
        }
        cudaError_t e = configure_mixed(mixed_cbc_dec_fn(nr), kSmemDec, mixed_cbc_dec_bit(nr));
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(cbc_fn(nr, true), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kSmemEnc);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(cbc_fn(nr, false), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemDec);
        if (e != cudaSuccess) return e;
        for (int lanes : {2, 4}) {
            e = cudaFuncSetAttribute(cbc_enc_split_fn(nr, lanes), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemEnc);
            if (e != cudaSuccess) return e;
        }
        for (bool permute : {false, true}) {
            e = cudaFuncSetAttribute(cbc_enc_staged_fn(nr, permute), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmemEncStaged);
            if (e != cudaSuccess) return e;
        }
        e = cudaFuncSetAttribute(cbc_enc_tma_fn(nr), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemEncTma);
        if (e != cudaSuccess) return e;
        for (int dir = 0; dir < 2; dir++) {
            if (!cts_fn(nr, dir)) continue;  // there is no XTS-AES-192
            e = cudaFuncSetAttribute(cts_fn(nr, dir), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cts_smem(dir));
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
    const bool usable = (g_mixed_usable.load() & mixed_bit(nr, dir, tweak)) != 0;
    const uint32_t spans = usable ? mix_spans(p.cta_chunks, nr, dir, tweak, tweak ? p.bps : 32, p.link != 0) : 0;
    if (spans) {
        MixParams mp;
        mp.b = p;
        mp.spans = spans;
        plane_masks(mp.masks, p.rk, nr);
        return launch(mixed_fn(nr, dir, tweak), grid, kMixThreads, mixed_smem(dir), s, mp);
    }
    return launch(fn, grid, kBulkThreads, bulk_smem(dir, tweak), s, p);
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
    num_sms = cbc_dec_sms(num_sms, p.bpp, p.npages * p.bpp * 16, p.link != 0);
    const bool in_place = p.src == p.dst;
    const uint64_t items = in_place ? p.npages : (p.npages * p.bpp + 31) / 32;
    const int grid = in_place ? (int)std::min<uint64_t>(items, num_sms) : grid_for_chunks(items, num_sms);
    if (items / grid >= 0xffffffffull) return cudaErrorInvalidValue;
    q.cta_items = (uint32_t)(items / grid);
    q.cta_rest = (uint32_t)(items % grid);
    const bool usable = !in_place && (g_mixed_usable.load() & mixed_cbc_dec_bit(nr)) != 0;
    const uint32_t spans = usable ? mix_spans(q.cta_items, nr, 1, false, p.bpp, p.link != 0) : 0;
    if (spans) {
        MixCbcParams mp;
        mp.c = q;
        mp.spans = spans;
        plane_masks(mp.masks, q.rk, nr);
        return launch(mixed_cbc_dec_fn(nr), grid, kMixThreads, kSmemDec, s, mp);
    }
    return launch(fn, grid, kBulkThreads, kSmemDec, s, q);
}

cudaError_t launch_xts_cts(const CtsParams& p, int nr, int dir, int num_sms, cudaStream_t s) {
    auto fn = cts_fn(nr, dir);
    if (!fn) return cudaErrorInvalidValue;
    CtsParams q = p;
    // a CTA per SM from four 32-block chunks each, and never less than a unit
    const uint64_t chunks = (p.units * (p.du / 16) + 31) / 32;
    const int grid = (int)std::min<uint64_t>(p.units, grid_for_chunks(chunks, num_sms));
    q.cta_units = p.units / grid;
    q.cta_rest = (uint32_t)(p.units % grid);
    return launch(fn, grid, kCtsThreads, cts_smem(dir), s, q);
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
    const uint64_t sms = (uint64_t)(num_sms > 0 ? num_sms : 1);
    const int lanes = cbc_enc_lanes(p.npages, p.bpp, nr, sms, p.link != 0);
    if (lanes > 1) {
        auto fn = cbc_enc_split_fn(nr, lanes);
        if (!fn) return cudaErrorInvalidValue;
        const uint64_t teams = (p.npages + 32 / lanes - 1) / (32 / lanes);
        return launch(fn, (int)cbc_enc_split_ctas(teams, sms), kCbcSplitThreads, kSmemEnc, s, p);
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
            return launch(fn, grid, warps * 32, kSmemEncTma, s, t);
        }
    }
    if (p.bpp % kStageBlocks == 0) {
        auto fn = cbc_enc_staged_fn(nr, p.npages <= 192 * sms);
        if (!fn) return cudaErrorInvalidValue;
        const int grid = (int)(groups < (uint64_t)num_sms ? (groups ? groups : 1) : num_sms);
        const int warps = cbc_enc_staged_warps(groups, num_sms);
        return launch(fn, grid, warps * 32, kSmemEnc + warps * kStageWarpSmem, s, p);
    }
    auto fn = cbc_fn(nr, true);
    if (!fn) return cudaErrorInvalidValue;
    // a 32-page group is a heavy work item (32 chains of whole pages): give
    // every SM work as soon as there are as many groups as SMs
    const int grid = (int)(groups < (uint64_t)num_sms ? (groups ? groups : 1) : num_sms);
    return launch(fn, grid, kBulkThreads, kSmemEnc, s, p);
}

}  // namespace kgpu
