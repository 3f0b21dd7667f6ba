// Device-side building blocks shared by the kernels: shared-memory table layout, the
// word-strided CRC chain, GF(2) products, team barriers and small load/store helpers.
//
// Work unit: a "team" of warps owns one 16 KiB tile at a time (eight warps in the decode kernel and the
// checksum of smaller caches, four in the encode kernel, one in the checksum of large caches).  The
// tile is seen as 128 rows of 128 bytes; a warp owns 16, 32 or all 128 consecutive rows and lane l owns
// the 32-bit word l of each of those rows.  A lane therefore walks words that are exactly 128 bytes
// apart, which makes its CRC contribution a Horner chain with ONE fixed multiplier
// (x^1024, table G); the lane's place inside the row and the warp's place inside the tile
// are folded in once per tile with two small nibble tables (NK, NW).
//
// Table lookups are the inner loop (one per byte), so their address arithmetic is reduced to one
// instruction, and to one that does not queue up with the rest: an entry of a table is 128 bytes and
// holds one copy per lane (lane l only ever touches bank l: no bank conflicts on data-dependent
// indices), so the address base + 128 * byte + 4 * lane is the dot product of the word's four bytes
// with a vector that picks one of them times 128 (dp4a).  That instruction runs on the multiplier's
// pipe.  The XORs, shifts, permutes and logic of everything else here share the other integer pipe,
// which is what these kernels fill first (measured, warp instructions per cycle and SM: permutes and
// logic together 2.0, dp4a and logic together 3.9).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "wm_tables.h"

namespace wm {

constexpr uint32_t kTile = 16384;
constexpr uint32_t kTeamThreads = 256;
constexpr uint32_t kShare = 2048;           // sixteen rows of a tile: what a warp holds, 16 words per lane
constexpr uint32_t kWordsPerLane = 16;
// Dynamic shared memory every table-using kernel asks for: the 144 KiB image and 81 KiB for stages and
// control blocks.  227 KiB is the per-block maximum for static and dynamic shared memory together;
// the kernels' static part is below 1 KiB.
constexpr uint32_t kDynSmem = kImgBytes + 0x14400;

struct Smem {
    uint32_t L;                  // shared-window address of the image + lane * 4
    const uint32_t* NW;          // warp-position nibble tables [8][8][16]
    unsigned char* free; uint32_t free_bytes;    // what is left behind the image
    bool ok;

    // carve `bytes` (multiple of 16) from the free space; nullptr when it does not fit
    __device__ unsigned char* take(uint32_t bytes)
    {
        if (free_bytes < bytes) { ok = false; return nullptr; }
        unsigned char* p = free;
        free += bytes; free_bytes -= bytes;
        return p;
    }
};

// Put the table image into shared memory (whole block; ends with __syncthreads).  A block fetches
// 24 KiB and makes the lanes' copies of G itself: fetching the finished image, 144 KiB for each of
// 148 blocks at once, is 21 MB out of L2 in front of every kernel, and the caches that are small
// enough to notice consist of such kernels.
__device__ __forceinline__ Smem setup_smem(unsigned char* smem, const Tables* __restrict__ tab)
{
    Smem s;
    s.ok = true;
    s.free = smem + kImgBytes; s.free_bytes = kDynSmem - kImgBytes;
    const uint32_t lane = threadIdx.x & 31u;
    uint4* dst = reinterpret_cast<uint4*>(smem);
    for (uint32_t e0 = (threadIdx.x / 32u) * 32u; e0 < 1024u; e0 += blockDim.x) {      // 32 entries per warp
        const uint32_t x = (&tab->G[0][0])[e0 + lane];
#pragma unroll
        for (uint32_t j = 0; j < 8u; j++) {            // four entries of 128 bytes at a time
            const uint32_t v = __shfl_sync(0xFFFFFFFFu, x, 4u * j + lane / 8u);
            dst[(e0 + 4u * j) * (kImgEntry / 16u) + lane] = make_uint4(v, v, v, v);
        }
    }
    const uint4* nk = reinterpret_cast<const uint4*>(&tab->NK[0][0][0]);
    for (uint32_t i = threadIdx.x; i < (kImgBytes - kImgNK) / 16u; i += blockDim.x) dst[kImgNK / 16u + i] = nk[i];
    uint32_t* nw = reinterpret_cast<uint32_t*>(s.take(8 * 8 * 16 * 4));
    if (nw) {
        const uint32_t* gNW = &tab->NW[0][0][0];
        for (uint32_t i = threadIdx.x; i < 8 * 8 * 16; i += blockDim.x) nw[i] = gNW[i];
    }
    s.NW = nw;
    s.L = (uint32_t)__cvta_generic_to_shared(smem) + lane * 4u;
    __syncthreads();
    return s;
}

// A value that is the same in every lane, told to the compiler: a warp reduction's result lives in a
// uniform register, arithmetic on it leaves the lanes' pipe alone and branches on it need no
// reconvergence bookkeeping.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __reduce_min_sync(0xFFFFFFFFu, v); }

template <int OFF>
__device__ __forceinline__ uint32_t lds_off(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}

// Loads of data that other threads or the copy engine write (stages, team control blocks),
// addressed by 32-bit shared-window addresses so that the address arithmetic stays in 32 bits.
// volatile: they keep their place relative to the barriers and mbarrier waits around them.
template <int OFF>
__device__ __forceinline__ uint32_t lds_now(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ uint2 lds_now_v2(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2+%3];" : "=r"(v.x), "=r"(v.y) : "r"(addr), "n"(OFF));
    return v;
}
__device__ __forceinline__ uint32_t lds_now_u16(uint32_t addr)
{
    uint32_t v;
    asm volatile("{\n\t.reg .u16 t;\n\tld.shared.u16 t, [%1];\n\tcvt.u32.u16 %0, t;\n\t}" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds_now_u8(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// Look-ups in tables that do not change once they are set up (no volatile: the compiler may place them)
__device__ __forceinline__ uint32_t lds_tab_u8(uint32_t addr)
{
    uint32_t v;
    asm("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds_tab_u16(uint32_t addr)
{
    uint32_t v;
    asm("{\n\t.reg .u16 t;\n\tld.shared.u16 t, [%1];\n\tcvt.u32.u16 %0, t;\n\t}" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_now(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Programmatic dependent launch.  Every call enqueues a short chain of kernels; each is launched with
// permission to start before its predecessor on the stream has finished (the first one too: its
// predecessor is the caller's or the previous call's last kernel).  It then
// sets up what does not depend on the predecessor (tables into shared memory, allocations) and
// waits here; the wait returns once the predecessor has completed and its writes are visible.
// Every block of such a kernel must pass the wait before it exits or reads anything the chain
// produced.  A kernel tells the scheduler that its successor may be brought in with
// grid_dep_launch (the successor's blocks take SM resources as they become free).
// Such a kernel's life begins before its predecessor has written all that it reads, and the read-only
// data path wants memory that does not change in a kernel's whole life.  So whatever a predecessor may
// still be writing (for a call's first kernel: everything the caller hands in; behind it, what the chain
// itself writes) is read through plain pointers or __ldcg, never through `const __restrict__`
// parameters or __ldg.  A chain's first kernel waits before it lets the second in, so the second and all
// behind it find the caller's data complete when they start.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void team_bar(uint32_t team)
{
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(kTeamThreads) : "memory");
}

// One chain step: (state ^ word) advanced over 128 bytes.
__device__ __forceinline__ uint32_t chain_step(const Smem& S, uint32_t x)
{
    const uint32_t a = lds_off<0 * kImgTable>(__dp4a(x, kImgEntry, S.L));
    const uint32_t b = lds_off<1 * kImgTable>(__dp4a(x, kImgEntry << 8, S.L));
    const uint32_t c = lds_off<2 * kImgTable>(__dp4a(x, kImgEntry << 16, S.L));
    const uint32_t d = lds_off<3 * kImgTable>(__dp4a(x, kImgEntry << 24, S.L));
    return a ^ b ^ c ^ d;
}

// Lane finish: x advanced over 128 - 4*lane bytes (eight nibble lookups; an odd nibble is 16 times its
// value in its byte, so its entry's place is 8 times that).
template <int N>
__device__ __forceinline__ uint32_t nibble_entry(const Smem& S, uint32_t xe, uint32_t xo)
{
    return lds_off<kImgNK + N * kImgNibble>((N & 1) ? __dp4a(xo, (kImgEntry / 16u) << (8 * (N / 2)), S.L)
                                                    : __dp4a(xe, kImgEntry << (8 * (N / 2)), S.L));
}
__device__ __forceinline__ uint32_t lane_finish(const Smem& S, uint32_t x)
{
    const uint32_t xe = x & 0x0F0F0F0Fu, xo = x & 0xF0F0F0F0u;
    return nibble_entry<0>(S, xe, xo) ^ nibble_entry<1>(S, xe, xo) ^ nibble_entry<2>(S, xe, xo) ^ nibble_entry<3>(S, xe, xo) ^
           nibble_entry<4>(S, xe, xo) ^ nibble_entry<5>(S, xe, xo) ^ nibble_entry<6>(S, xe, xo) ^ nibble_entry<7>(S, xe, xo);
}

// CRC state (zero start) of a warp's 2048-byte block from the 16 words each lane holds.
__device__ __forceinline__ uint32_t warp_block_digest(const Smem& S, const uint32_t (&w)[kWordsPerLane])
{
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < 15; i++) s = chain_step(S, s ^ w[i]);
    return __reduce_xor_sync(0xFFFFFFFFu, lane_finish(S, s ^ w[15]));
}

// Place a warp's block digest inside the tile: advance over 2048*(7 - warp) bytes.  Returns the
// warp's contribution to the tile digest in every lane.
__device__ __forceinline__ uint32_t warp_place(const Smem& S, uint32_t digest, uint32_t warp, uint32_t lane)
{
    uint32_t v = 0;
    if (lane < 8) v = S.NW[(warp * 8 + lane) * 16 + ((digest >> (4 * lane)) & 15u)];
    return __reduce_xor_sync(0xFFFFFFFFu, v);
}

// The tile's digest from its eight warps' block digests (one warp, the result in every lane): lane l
// places nibbles 2 (l mod 4) and the next of warp l / 4's digest.  In the codec kernels one warp does
// this for the team, a step later, where each warp placing its own digest is a look-up, two reductions
// and their wait in every warp.  wdig_s: shared-window address of the eight digests.
__device__ __forceinline__ uint32_t place_warp_digests(const Smem& S, uint32_t wdig_s, uint32_t lane)
{
    const uint32_t d = lds_now<0>(wdig_s + (lane & ~3u));
    const uint32_t n = 2u * (lane & 3u);                     // table row 8 (lane / 4) + n = 2 lane
    const uint32_t at = S.L - 4u * lane + kImgBytes + 128u * lane;       // (the position tables stand behind the image)
    const uint32_t b = d >> (4u * n);
    const uint32_t v = lds_off<0>(at + 4u * (b & 15u)) ^ lds_off<64>(at + 4u * ((b >> 4) & 15u));
    return __reduce_xor_sync(0xFFFFFFFFu, v);
}

// The same for a tile's four warps of 4096 bytes (rows 32 w ..): lane l places nibble l mod 8 of warp l / 8's digest.
__device__ __forceinline__ uint32_t place_team4_digests(const Smem& S, uint32_t wdig_s, uint32_t lane)
{
    const uint32_t w = lane >> 3, n = lane & 7u;
    const uint32_t d = lds_now<0>(wdig_s + 4u * w);
    // (advancing over 4096 (3 - w) bytes is row 2 w + 1 of the tables for 2048-byte blocks)
    return __reduce_xor_sync(0xFFFFFFFFu, lds_off<0>(S.L - 4u * lane + kImgBytes + 64u * (8u * (2u * w + 1u) + n) + 4u * ((d >> (4u * n)) & 15u)));
}

// ---- the same digest with small tables, for kernels that see a few hundred kilobytes ----
// Copying the 144 KiB lane-replicated image costs more than such a kernel's whole work.  Here
// the chain uses one copy of the four byte tables (4 KiB in shared memory; lookups may collide on a
// bank) and the two once-per-tile steps read the
// nibble tables straight from global memory.  Same result as warp_block_digest + warp_place.
__device__ __forceinline__ void load_small_chain_tables(uint32_t* sG, const Tables* __restrict__ tab)
{
    for (uint32_t i = threadIdx.x; i < 1024; i += blockDim.x) sG[i] = (&tab->G[0][0])[i];
    __syncthreads();
}
__device__ __forceinline__ uint32_t tile_digest_part_small(const uint32_t* sG, const Tables* __restrict__ tab,
                                                           const uint32_t (&w)[kWordsPerLane], uint32_t warp, uint32_t lane)
{
    uint32_t s = 0;
#pragma unroll
    for (int i = 0; i < 15; i++) {
        const uint32_t x = s ^ w[i];
        s = sG[x & 0xFFu] ^ sG[256u + ((x >> 8) & 0xFFu)] ^ sG[512u + ((x >> 16) & 0xFFu)] ^ sG[768u + (x >> 24)];
    }
    const uint32_t x = s ^ w[15];
    uint32_t r = 0;
#pragma unroll
    for (uint32_t n = 0; n < 8; n++)
        r ^= __ldg(&tab->NK[n][(x >> (4u * n)) & 15u][lane]);
    const uint32_t digest = __reduce_xor_sync(0xFFFFFFFFu, r);
    uint32_t v = 0;
    if (lane < 8) v = __ldg(&tab->NW[warp][lane][(digest >> (4 * lane)) & 15u]);
    return __reduce_xor_sync(0xFFFFFFFFu, v);
}

// Generic product of two residues (bitwise; used a handful of times per call).
__device__ __forceinline__ uint32_t mulmod_dev(uint32_t a, uint32_t b, uint32_t poly = kPolyReflected)
{
    uint32_t r = 0;
#pragma unroll 8
    for (int i = 0; i < 32; i++) {
        r ^= b & (0u - (a >> 31));
        a <<= 1;
        b = (b >> 1) ^ (poly & (0u - (b & 1u)));
    }
    return r;
}

// Advance a state over one tile (16384 bytes) with byte tables HT[4][256] (shared or global).
__device__ __forceinline__ uint32_t advance_tile(const uint32_t* HT, uint32_t s)
{
    return HT[s & 0xFF] ^ HT[256 + ((s >> 8) & 0xFF)] ^ HT[512 + ((s >> 16) & 0xFF)] ^ HT[768 + (s >> 24)];
}

__device__ __forceinline__ void st_stream_u32(void* p, uint32_t v)
{
    asm volatile("st.global.cs.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Shifts whose amount may be 32 (the result is then 0, as the hardware's shifts define it; in C
// a shift by the operand's width is undefined).
__device__ __forceinline__ uint32_t shl_clamp(uint32_t v, uint32_t n)
{
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}
__device__ __forceinline__ uint32_t shr_clamp(uint32_t v, uint32_t n)
{
    uint32_t r;
    asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ uint32_t max_u16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// ---- bulk (TMA) copies of whole tiles into shared memory, tracked by an mbarrier ----
// Loads that land in registers long before they are used tie up the warp's few scoreboards:
// every later shared-memory or global access that shares one waits for them, so "prefetching
// into registers" serialises instead of overlapping.  A bulk copy is issued by one thread,
// holds no registers while in flight, and its completion is observed on an mbarrier.
__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(a), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// One 16-byte aligned copy of `bytes` (multiple of 16) from global to shared memory; the
// mbarrier's pending byte count is raised first.  `policy`: an L2 cache policy or 0.
__device__ __forceinline__ void bulk_load(void* smem_dst, const void* gsrc, uint32_t bytes, unsigned long long* bar,
                                          uint64_t policy)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    if (policy)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                     ::"r"(d), "l"(gsrc), "r"(bytes), "r"(b), "l"(policy) : "memory");
    else
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(d), "l"(gsrc), "r"(bytes), "r"(b) : "memory");
}

// The same with both shared-memory places given by their 32-bit shared-window addresses.
__device__ __forceinline__ void bulk_load_at(uint32_t d, const void* gsrc, uint32_t bytes, uint32_t b, uint64_t policy)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    if (policy)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                     ::"r"(d), "l"(gsrc), "r"(bytes), "r"(b), "l"(policy) : "memory");
    else
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(d), "l"(gsrc), "r"(bytes), "r"(b) : "memory");
}

// The low 32 bits of the GPU's wall clock in nanoseconds (they wrap every 4.29 s).  Every
// device-side wait is bounded by TIME against the call's budget (Geo::wait_ns, two seconds unless
// the caller set another, never more than four), not by a number of polls: a block that shares
// the GPU with other work can be descheduled for a long time, and a poll count says nothing about
// how long that was.  Differences of two readings are taken modulo 2^32, which is exact for
// spans below the wrap.
__device__ __forceinline__ uint32_t now_ns()
{
    uint32_t t;
    asm volatile("mov.u32 %0, %%globaltimer_lo;" : "=r"(t));
    return t;
}

// Wait for the phase with the given parity to complete, for at most `budget_ns`.  Returns false
// when the time ran out.  try_wait suspends the thread in hardware until the phase completes or
// the time hint runs out, so a waiting warp does not burn issue slots that the other teams on
// the SM need.  (The waiting loop itself, wait_for_copy_at, follows the control block's definition.)
__device__ __forceinline__ uint32_t mbar_try(uint32_t bar_s, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar_s), "r"(parity), "r"(200000u) : "memory");
    return done;
}
// The same question without waiting at all; one arrival.
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar_s, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done) : "r"(bar_s), "r"(parity) : "memory");
    return done;
}
__device__ __forceinline__ void mbar_arrive_at(uint32_t bar_s)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_s) : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_first()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// ---- tensor memory as a parking place for tiles in flight ----
// Each SM has 256 KB of tensor memory (128 lanes x 512 columns of 32 bits) next to its shared
// memory.  Nothing here multiplies matrices, so it is free, and it takes exactly the shape of
// what a team has to park: thread i of a warp owns lane 32 * (warp % 4) + i, and one
// instruction moves 16 consecutive columns between that lane and 16 registers.  A tile that has
// been measured waits there for its place in the wire image instead of being fetched again.
// The block allocates all 512 columns once (it is alone on its SM) and must free them before
// it exits.  All of these are warp-wide (.sync.aligned): every lane of the warp executes them.
__device__ __forceinline__ void tmem_alloc_all(uint32_t* smem_result)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(smem_result);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(a) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free_all(uint32_t taddr)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 registers -> 16 columns of this thread's lane, and back.  A store is waited for when the
// next one is issued and once more before the memory is handed back; its data is fetched two steps
// on, behind a wait of its own (tmem_wait_stores in front of the fetch) that finds it long done.
__device__ __forceinline__ void tmem_wait_stores() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_store16(uint32_t taddr, const uint32_t (&w)[16])
{
    tmem_wait_stores();
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]),
                   "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15]) : "memory");
}
__device__ __forceinline__ void tmem_load16(uint32_t taddr, uint32_t (&w)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]),
                   "=r"(w[8]), "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15])
                 : "r"(taddr) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 bytes from global to shared memory without a register in between (both 16-byte aligned;
// past L1).  A thread that has issued some waits for its own with cp_async_wait_all.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A staged tile's words for this lane: word `lane` of rows 16*warp .. 16*warp+15 (conflict free).
__device__ __forceinline__ void read_staged_words(const unsigned char* stage, uint32_t warp, uint32_t lane,
                                                  uint32_t (&w)[16])
{
    const uint32_t* p = reinterpret_cast<const uint32_t*>(stage) + warp * 512u + lane;
#pragma unroll
    for (int i = 0; i < 16; i++) w[i] = p[i * 32];
}

// (the stage given by its 32-bit shared-window address)
__device__ __forceinline__ void read_staged_words_at(uint32_t stage_s, uint32_t warp, uint32_t lane, uint32_t (&w)[16])
{
    const uint32_t p = stage_s + 4u * (warp * 512u + lane);
    w[0] = lds_now<0>(p);     w[1] = lds_now<128>(p);   w[2] = lds_now<256>(p);   w[3] = lds_now<384>(p);
    w[4] = lds_now<512>(p);   w[5] = lds_now<640>(p);   w[6] = lds_now<768>(p);   w[7] = lds_now<896>(p);
    w[8] = lds_now<1024>(p);  w[9] = lds_now<1152>(p);  w[10] = lds_now<1280>(p); w[11] = lds_now<1408>(p);
    w[12] = lds_now<1536>(p); w[13] = lds_now<1664>(p); w[14] = lds_now<1792>(p); w[15] = lds_now<1920>(p);
}

// ---- the ragged last tile of a cache: `len` (1..16383) real bytes, stored raw ----
// One team handles it outside the kernels' loops, which then know full tiles only.  For the checksum
// it goes into the team's stage right-aligned in a virtual tile whose leading 16384 - len bytes are
// zero (leading zeros do not change a zero-start CRC state) and is read from there like any other
// tile.  When `first_in_chunk`, the chunk's first four bytes are complemented (the all-ones CRC
// init).  `tile` is four-byte aligned; no byte behind its end is read.  A thread takes sixteen
// words and has all of its loads under way together: the tile is one trip to memory long, where
// fetching its words one after the other, byte by byte, took 8 us more (decode of 8 MB: 36.8 us ->
// 28.7; 18.6 with what came after), which every call waited for at its end.
__device__ __forceinline__ void stage_ragged_tile(unsigned char* stage, const unsigned char* __restrict__ tile, uint32_t len,
                                                  bool first_in_chunk, uint32_t tt)
{
    const int32_t pad = (int32_t)(kTile - len);
    const uint32_t off = len & 3u;                     // (a virtual word starts at real byte 4 q - pad, off modulo four)
    const uint32_t* p = reinterpret_cast<const uint32_t*>(tile);
    uint32_t v[16];
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const int32_t rb = 4 * (int32_t)(tt + kTeamThreads * i) - pad;      // the word's first real byte
        const int32_t a = rb >> 2;
        uint32_t lo = 0, hi = 0;
        if (a >= 0) lo = __ldcg(p + a);
        if (off && a >= -1 && 4 * (a + 2) <= (int32_t)len) hi = __ldcg(p + a + 1);
        v[i] = __funnelshift_r(lo, hi, 8u * off);
    }
    if (off && tt == kTeamThreads - 1u) {              // the last word: its last bytes are not a whole word of the tile
        const uint32_t at = len & ~3u;
        for (uint32_t j = 0; j < off; j++) v[15] |= (uint32_t)__ldcg(tile + at + j) << (8u * (4u - off + j));
    }
#pragma unroll
    for (int i = 0; i < 16; i++) {
        const uint32_t q = tt + kTeamThreads * i;
        const int32_t rb = 4 * (int32_t)q - pad;
        if (first_in_chunk && rb > -4 && rb < 4)
            v[i] ^= rb < 0 ? 0xFFFFFFFFu << (8 * -rb) : 0xFFFFFFFFu >> (8 * rb);
        reinterpret_cast<uint32_t*>(stage)[q] = v[i];
    }
    // (the stage's next content comes by a bulk copy, which is another proxy)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The same tile's `len` bytes from one 16-byte aligned place to another, by a team's 256 threads.
__device__ __forceinline__ void copy_ragged_tile(unsigned char* __restrict__ dst, const unsigned char* __restrict__ src, uint32_t len,
                                                 uint32_t tt)
{
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        v[i] = make_uint4(0, 0, 0, 0);
        if (16u * (tt + kTeamThreads * i) + 16u <= len) v[i] = __ldcg(reinterpret_cast<const uint4*>(src) + tt + kTeamThreads * i);
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
        if (16u * (tt + kTeamThreads * i) + 16u <= len) reinterpret_cast<uint4*>(dst)[tt + kTeamThreads * i] = v[i];
    const uint32_t at = (len & ~15u) + tt;
    if (at < len) dst[at] = __ldcg(src + at);
}

// CRC32C of a short run computed byte by byte (chunks shorter than four bytes).
__device__ __forceinline__ uint32_t crc_bytewise(const uint32_t* T0, const unsigned char* p, uint32_t n)
{
    uint32_t crc = 0xFFFFFFFFu;
    for (uint32_t i = 0; i < n; i++) crc = T0[(crc ^ __ldcg(p + i)) & 0xFF] ^ (crc >> 8);
    return ~crc;
}

// Exclusive prefix of `v` over the threads of a 1024-thread block, in thread order, and the
// block's total.  s_part: 33 values of shared memory.  Block-wide (two barriers); one use per
// kernel, or a barrier between uses.  The kernels that scan a per-chunk array give every thread
// a run of consecutive chunks, so one such prefix does for any number of chunks.
template <typename T>
__device__ __forceinline__ T block_prefix(T v, T* s_part, T& total)
{
    const uint32_t lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    T incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const T o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    if (lane == 31) s_part[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const T p = s_part[lane];
        T pi = p;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const T o = __shfl_up_sync(0xFFFFFFFFu, pi, d);
            if (lane >= (uint32_t)d) pi += o;
        }
        s_part[lane] = pi - p;
        if (lane == 31) s_part[32] = pi;
    }
    __syncthreads();
    total = s_part[32];
    return s_part[warp] + incl - v;
}

}  // namespace wm
