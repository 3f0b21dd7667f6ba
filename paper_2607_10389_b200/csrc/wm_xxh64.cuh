// wm_checksum_xxh64: the 64-bit xxHash of every chunk, as a checksum option beside the CRC.
// Part of the one translation unit wm_kernels.cu (included there, in this order).
//
// XXH64 takes its input in 32-byte stripes into four accumulators; lane k of a stripe feeds
// accumulator k through  acc = rotl(acc + in * P2, 31) * P1,  a serial chain over the whole chunk
// (digests of pieces cannot be combined, unlike a CRC).  So a chunk offers four threads of work and
// the parallelism is across chunks; a warp holds eight of them.  There are two kernels.
//   k_xxh64        a warp loads its chunks' data into registers two batches ahead and walks the
//                  chains.  With many chunks (64 KiB each, say) there are chains enough to cover
//                  the loads and the products, and it runs at the memory rate (6.2 TB/s).
//   k_xxh64_paced  for few chunks, where the latency of one chain step bounds the call: a chain warp
//                  has a scheduler to itself and does nothing but chain steps, other warps bring the
//                  data in and take the products.
#pragma once
#include "wm_xxh64_plan.h"

namespace wm {

constexpr unsigned long long kXP1 = 0x9E3779B185EBCA87ull, kXP2 = 0xC2B2AE3D27D4EB4Full, kXP3 = 0x165667B19E3779F9ull,
                             kXP4 = 0x85EBCA77C2B2AE63ull, kXP5 = 0x27D4EB2F165667C5ull;

__device__ __forceinline__ unsigned long long x_rotl(unsigned long long v, int r) { return (v << r) | (v >> (64 - r)); }
__device__ __forceinline__ unsigned long long x_round(unsigned long long acc, unsigned long long in)
{
    return x_rotl(acc + in * kXP2, 31) * kXP1;
}
__device__ __forceinline__ unsigned long long x_merge(unsigned long long h, unsigned long long v)
{
    return (h ^ x_round(0ull, v)) * kXP1 + kXP4;
}

// The four accumulators merged, the bytes behind the last whole stripe, the avalanche.
__device__ __forceinline__ unsigned long long x_finish(const unsigned char* base, uint64_t len, unsigned long long seed,
                                                       unsigned long long v1, unsigned long long v2, unsigned long long v3,
                                                       unsigned long long v4)
{
    unsigned long long h;
    if (len >= 32u) {
        h = x_rotl(v1, 1) + x_rotl(v2, 7) + x_rotl(v3, 12) + x_rotl(v4, 18);
        h = x_merge(h, v1); h = x_merge(h, v2); h = x_merge(h, v3); h = x_merge(h, v4);
    } else {
        h = seed + kXP5;
    }
    h += len;
    const unsigned char* t = base + (len & ~31ull);
    uint32_t left = (uint32_t)len & 31u;
    while (left >= 8u) {
        h = x_rotl(h ^ x_round(0ull, *reinterpret_cast<const unsigned long long*>(t)), 27) * kXP1 + kXP4;
        t += 8; left -= 8u;
    }
    if (left >= 4u) {
        h = x_rotl(h ^ ((unsigned long long)*reinterpret_cast<const uint32_t*>(t) * kXP1), 23) * kXP2 + kXP3;
        t += 4; left -= 4u;
    }
    while (left) { h = x_rotl(h ^ ((unsigned long long)*t * kXP5), 11) * kXP1; t++; left--; }
    h ^= h >> 33; h *= kXP2; h ^= h >> 29; h *= kXP3; h ^= h >> 32;
    return h;
}

constexpr int kXBatch = 32;       // stripes per batch of loads

__global__ void __launch_bounds__(32)
k_xxh64(const unsigned char* __restrict__ cache, uint64_t nbytes, uint32_t chunk_bytes, uint32_t n_chunks,
        unsigned long long seed, unsigned long long* __restrict__ out)
{
    const uint32_t c = 8u * blockIdx.x + threadIdx.x / 4u, k = threadIdx.x & 3u;       // (a chunk's number: 4 c need not fit 32 bits)
    const bool live = c < n_chunks;                     // (a quad is live or dead as a whole)
    const unsigned char* base = cache;
    uint64_t len = 0;
    if (live) {
        base = cache + (uint64_t)c * chunk_bytes;
        const uint64_t left = nbytes - (uint64_t)c * chunk_bytes;
        len = left < chunk_bytes ? left : chunk_bytes;
    }
    const uint64_t stripes = len / 32u;
    unsigned long long v = k == 0u ? seed + kXP1 + kXP2 : k == 1u ? seed + kXP2 : k == 2u ? seed : seed - kXP1;
    // (the cache is 16-byte aligned and chunks are multiples of 16 KiB: aligned 8-byte loads)
    const unsigned long long* p = reinterpret_cast<const unsigned long long*>(base) + k;
    unsigned long long a[kXBatch], b[kXBatch];
    uint64_t s = 0;
    if (stripes >= (uint64_t)kXBatch) {
#pragma unroll
        for (int i = 0; i < kXBatch; i++) a[i] = __ldcs(p + 4u * i) * kXP2;
        // two batches per turn: while one is folded into the accumulator the other is on its way
        while (s + 2u * kXBatch <= stripes) {
#pragma unroll
            for (int i = 0; i < kXBatch; i++) b[i] = __ldcs(p + 4u * (s + kXBatch + i)) * kXP2;
#pragma unroll
            for (int i = 0; i < kXBatch; i++) v = x_rotl(v + a[i], 31) * kXP1;
            s += kXBatch;
            if (s + 2u * kXBatch <= stripes) {
#pragma unroll
                for (int i = 0; i < kXBatch; i++) a[i] = __ldcs(p + 4u * (s + kXBatch + i)) * kXP2;
#pragma unroll
                for (int i = 0; i < kXBatch; i++) v = x_rotl(v + b[i], 31) * kXP1;
                s += kXBatch;
            } else {
#pragma unroll
                for (int i = 0; i < kXBatch; i++) a[i] = b[i];
            }
        }
        // a[] holds the batch that starts at s
#pragma unroll
        for (int i = 0; i < kXBatch; i++) v = x_rotl(v + a[i], 31) * kXP1;
        s += kXBatch;
    }
    for (; s < stripes; s++) v = x_round(v, __ldcs(p + 4u * s));

    // the quad's four accumulators to its first thread; merge, tail, avalanche
    const uint32_t q0 = threadIdx.x & ~3u;
    const unsigned long long v1 = __shfl_sync(0xFFFFFFFFu, v, q0), v2 = __shfl_sync(0xFFFFFFFFu, v, q0 + 1u),
                             v3 = __shfl_sync(0xFFFFFFFFu, v, q0 + 2u), v4 = __shfl_sync(0xFFFFFFFFu, v, q0 + 3u);
    if (!live || k != 0u) return;
    out[c] = x_finish(base, len, seed, v1, v2, v3, v4);
}

// ---- few chunks: one warp walks the chains, the others feed it
constexpr uint32_t kXSeg = 64;                          // stripes of every chunk in one slot of the ring
constexpr uint32_t kXRowBytes = 32u * kXSeg;
constexpr uint32_t kXPitch = kXRowBytes + 32u;          // (rows 32 bytes apart modulo 128: the chains' reads meet no bank twice)
constexpr uint32_t kXSlot = kXRows * kXPitch;
constexpr uint32_t kXSlots = 3;                         // slots of a ring (4: 13.4 ns a step, 3: 13.1)
constexpr uint32_t kXRing = kXSlots * kXSlot;
constexpr uint32_t kXFeeders = 4;                       // warps that bring the data in and multiply it
constexpr uint32_t kXSets = 3;                          // slots' data that a feeder has under way in registers
constexpr uint32_t kXThreads = 512;                     // (warps 0, 1: chains; 2, 3, 6, 7 and 10, 11, 14, 15: their feeders, on the other two schedulers)

// A warp's wait for a phase of a barrier in shared memory, for at most the budget; the answer is the
// same in every lane.  The call has no result record to say that it failed, and it cannot fail: when a
// wait runs out, the block's warps leave the ring (`fail`) and the chain warp hashes its chunks with
// loads of its own (x_walk).
__device__ __forceinline__ bool x_wait(uint32_t bar, uint32_t parity, uint32_t budget_ns, volatile uint32_t* fail)
{
    bool ok = mbar_try(bar, parity) != 0u;
    if (!ok) {
        const uint32_t t0 = now_ns();
        do {
            ok = mbar_try(bar, parity) != 0u;
        } while (!ok && *fail == 0u && now_ns() - t0 <= budget_ns);
    }
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (!ok) *fail = 1u;
    return ok;
}
// One step of a chain: s' = rotl(s, 31) * P1 + x.  Written out in 32-bit halves: behind the rotation
// (two funnel shifts) stand one wide product with x as its addend and, beside it, the two products
// that only reach the high half; one add joins them.  23 cycles a step, where the plain formula
// takes 28 as it is compiled.
__device__ __forceinline__ unsigned long long x_step(unsigned long long s, unsigned long long x)
{
    const uint32_t p1lo = (uint32_t)kXP1, p1hi = (uint32_t)(kXP1 >> 32);
    const uint32_t lo = (uint32_t)s, hi = (uint32_t)(s >> 32);
    const uint32_t rl = __funnelshift_r(hi, lo, 1), rh = __funnelshift_r(lo, hi, 1);       // rotl 31 = halves swapped, one to the right
    unsigned long long w;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(w) : "r"(rl), "r"(p1lo), "l"(x));
    const uint32_t b = rh * p1lo + rl * p1hi;
    return (unsigned long long)(uint32_t)w | ((unsigned long long)((uint32_t)(w >> 32) + b) << 32);
}

// x_step(x_before(v), x) is v + x: the state in front of a chain's first stripe.
constexpr unsigned long long x_inverse(unsigned long long p)      // modulo 2^64 (Newton; p odd)
{
    unsigned long long r = p;
    for (int i = 0; i < 6; i++) r *= 2u - p * r;
    return r;
}
constexpr unsigned long long kXP1Inverse = x_inverse(kXP1);
__device__ __forceinline__ unsigned long long x_before(unsigned long long v) { return x_rotl(v * kXP1Inverse, 33); }

__device__ __forceinline__ void x_load1(unsigned long long& x, uint32_t a) { asm volatile("ld.shared.u64 %0, [%1];" : "=l"(x) : "r"(a)); }

// Accumulator k of a chunk from its start value, without the ring: sixteen stripes' loads at a time.  The
// rare path of a wait that ran out; kept out of line.
__device__ __noinline__ unsigned long long x_walk(unsigned long long v, const unsigned char* base, uint32_t stripes, uint32_t k)
{
    const unsigned long long* p = reinterpret_cast<const unsigned long long*>(base) + k;
    for (uint32_t i = 0; i < stripes; i += 16u) {
        unsigned long long in[16];
#pragma unroll
        for (uint32_t j = 0; j < 16u; j++) in[j] = i + j < stripes ? p[4ull * (i + j)] : 0ull;
#pragma unroll
        for (uint32_t j = 0; j < 16u; j++)
            if (i + j < stripes) v = x_round(v, in[j]);
    }
    return v;
}

// One block at a time on an SM: its 512 threads' registers (126 each) leave no room for a second one; with 64
// or fewer two would fit, and four chains would meet on two schedulers.  A block takes `rows` chunks, the last one what
// is left: up to eight by one chain warp, up to sixteen by two (the first has rows0 of them), each with a ring and feeders
// of its own.  The chains stand on schedulers of their own: a second chain on the same one costs both of them.
// What bounds it is the latency of a step, 23 cycles (11.7 ns); it takes 13.1 ns one chain to an SM and 13.2 with
// two (1.67 GB in 1 MiB chunks 605 -> 432 us, 2.48 GB 640 -> 434).  Before, a block had eight chunks and one chain,
// two such blocks could stand on an SM, and wherever the second one's warps came to stand they shared the
// first one's scheduler: 14.8 ns alone, 18.4 together.
__global__ void __launch_bounds__(kXThreads, 1)
k_xxh64_paced(const unsigned char* __restrict__ cache, uint64_t nbytes, uint32_t chunk_bytes, uint32_t n_chunks,
              unsigned long long seed, unsigned long long* __restrict__ out, uint32_t rows, uint32_t rows0, uint32_t wait_ns, uint32_t inject)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_full[2][kXSlots], s_empty[2][kXSlots];
    __shared__ uint32_t s_fail;
    const uint32_t warp = threadIdx.x / 32u, lane = threadIdx.x % 32u;
    const uint32_t half = (warp & 2u) ? warp >> 3 : warp & 1u;           // whose chain this warp belongs to
    const uint32_t c0 = blockIdx.x * rows + (half ? rows0 : 0u), my_rows = half ? rows - rows0 : rows0;      // the chain's chunks
    if (threadIdx.x < 2u * kXSlots) {
        // (test hook: a slot waits for one feeder more than there are)
        mbar_init(&s_full[0][threadIdx.x], kXFeeders + ((inject & kInjectNoCopy) ? 1u : 0u));
        mbar_init(&s_empty[0][threadIdx.x], 1);
        s_fail = 0;
    }
    __syncthreads();
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem) + half * kXRing;
    const uint32_t full = (uint32_t)__cvta_generic_to_shared(s_full[half]), empty = (uint32_t)__cvta_generic_to_shared(s_empty[half]);
    auto length = [&](uint32_t row) -> uint32_t {        // bytes of the chain's row-th chunk (0: there is none)
        const uint32_t c = c0 + row;
        if (row >= my_rows || c >= n_chunks) return 0u;
        const uint64_t left = nbytes - (uint64_t)c * chunk_bytes;
        return left < chunk_bytes ? (uint32_t)left : chunk_bytes;
    };
    const uint32_t n_seg = (length(0u) / 32u + kXSeg - 1u) / kXSeg;      // (the first chunk is the longest)

    if (warp & 2u) {
        // ---- the warps that feed the ring, two chunks each: sixteen lanes take 256 consecutive bytes of
        // one chunk at a time, straight into registers, kXSets slots ahead; the products go to the ring.
        // (Copied into the ring first and multiplied there, every byte passed through shared memory four
        // times, and that was what two blocks on one SM shared: 18.4 ns a step.)
        const uint32_t feeder = (warp & 1u) + ((warp >> 2) & 1u) * 2u;
        const uint32_t row = 2u * feeder + lane / 16u, col = 16u * (lane % 16u);
        const uint32_t mine = ring + row * kXPitch + col;
        constexpr uint32_t kUnits = kXRowBytes / 256u;   // 16-byte pieces of a slot per lane
        const uint32_t whole = length(row) & ~31u;       // bytes in whole stripes
        const unsigned char* const p = cache + (uint64_t)(whole ? c0 + row : 0u) * chunk_bytes + col;
        ulonglong2 in[kXSets][kUnits];
        auto fetch = [&](ulonglong2 (&x)[kUnits], uint32_t s) {
            const uint32_t at = s * kXRowBytes;
#pragma unroll
            for (uint32_t i = 0; i < kUnits; i++)
                x[i] = at + 256u * i + col < whole ? __ldcs(reinterpret_cast<const ulonglong2*>(p + at + 256u * i)) : make_ulonglong2(0ull, 0ull);
        };
#pragma unroll
        for (uint32_t j = 0; j < kXSets; j++) fetch(in[j], j);
        uint32_t slot = 0, parity = 1u;                  // (a barrier's phase before its first counts as complete)
        for (uint32_t s0 = 0; s0 < n_seg; s0 += kXSets) {
#pragma unroll
            for (uint32_t j = 0; j < kXSets; j++) {
                const uint32_t s = s0 + j;
                if (s >= n_seg) return;
                if (!x_wait(empty + 8u * slot, parity, wait_ns, &s_fail)) return;
                const uint32_t a = mine + slot * kXSlot;
#pragma unroll
                for (uint32_t i = 0; i < kUnits; i++)
                    asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(a + 256u * i), "l"(in[j][i].x * kXP2), "l"(in[j][i].y * kXP2) : "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_at(full + 8u * slot);
                fetch(in[j], s + kXSets);
                slot = slot + 1u == kXSlots ? 0u : slot + 1u;
                if (slot == 0u) parity ^= 1u;
            }
        }
        return;
    }
    if (warp > 1u) return;

    // ---- the chains: lane 4 r + k is accumulator k of chunk r of the eight
    const uint32_t k = lane & 3u, row = lane >> 2;
    const uint32_t mine = ring + row * kXPitch + 8u * k;
    const uint32_t c = c0 + row;
    const uint32_t len = length(row), stripes = len / 32u;
    // A segment in whose midst a chunk ends (only the cache's last chunk can) is walked with a test
    // per stripe.  Behind its chunk's end a chain runs on with whatever lies in its row, its result
    // having been put aside.
    const uint32_t uneven = __ballot_sync(0xFFFFFFFFu, stripes % kXSeg != 0u);
    const uint32_t odd_seg = uneven ? __shfl_sync(0xFFFFFFFFu, stripes, __ffs(uneven) - 1) / kXSeg : 0xFFFFFFFFu;
    // the state is the accumulator with the next product already added; the last step adds 0
    unsigned long long v = k == 0u ? seed + kXP1 + kXP2 : k == 1u ? seed + kXP2 : k == 2u ? seed : seed - kXP1;
    unsigned long long s = x_before(v), at_end = 0ull;
    unsigned long long x0[16], x1[16];
    // sixteen steps, the loads of the next sixteen between them (in one run in front of the steps they held the
    // chain up)
    auto steps = [&](const unsigned long long (&x)[16], unsigned long long (&next)[16], uint32_t from) {
#pragma unroll
        for (int i = 0; i < 16; i++) {
            s = x_step(s, x[i]);
            x_load1(next[i], from + 32u * i);
        }
    };
    const uint32_t end_seg = (stripes + kXSeg - 1u) / kXSeg;         // of this lane's chunk
    bool ok = n_seg == 0u || x_wait(full, 0u, wait_ns, &s_fail);
    uint32_t slot = 0, parity = 0, a = mine;             // of segment g
    uint32_t n_slot = 0, n_parity = 0, n_a = 0;          // of the one behind it
    auto look_ahead = [&]() {
        const bool wrap = slot + 1u == kXSlots;
        n_slot = wrap ? 0u : slot + 1u;
        n_parity = parity ^ (wrap ? 1u : 0u);
        n_a = wrap ? mine : a + kXSlot;
    };
    auto done = [&](uint32_t g) {                        // with segment g
        if (end_seg == g + 1u) at_end = s;
        __syncwarp();
        if (lane == 0) mbar_arrive_at(empty + 8u * slot);
        slot = n_slot; parity = n_parity; a = n_a;
    };
    for (uint32_t g = 0; g < n_seg && ok;) {
        if (g == odd_seg) {
            look_ahead();
            for (uint32_t i = 0; i < kXSeg; i++) {
                unsigned long long x;
                x_load1(x, a + 32u * i);
                const unsigned long long n = x_step(s, x);
                if (g * kXSeg + i < stripes) s = n;
            }
            if (g + 1u < n_seg) ok = x_wait(full + 8u * n_slot, n_parity, wait_ns, &s_fail);
            done(g++);
            continue;
        }
        const uint32_t g1 = g < odd_seg ? min(odd_seg, n_seg) : n_seg;       // the segments up to here have no chunk's end in their midst
#pragma unroll
        for (int i = 0; i < 16; i++) x_load1(x0[i], a + 32u * i);
        for (; g < g1 && ok; g++) {
            // whether the next segment is there is asked while this one's third quarter is still to be walked,
            // and its first words are fetched during the last: nothing waits at the seam.  (Behind the last
            // segment they are fetched from a slot that holds something else, and not used.)
            look_ahead();
            steps(x0, x1, a + 512u);
            steps(x1, x0, a + 1024u);
            const uint32_t ready = g + 1u < n_seg ? mbar_test(full + 8u * n_slot, n_parity) : 1u;
            steps(x0, x1, a + 1536u);
            if (!__all_sync(0xFFFFFFFFu, ready != 0u)) ok = x_wait(full + 8u * n_slot, n_parity, wait_ns, &s_fail);
            steps(x1, x0, n_a);
            done(g);
        }
    }
    if (!ok) v = x_walk(v, cache + (uint64_t)(stripes ? c : 0u) * chunk_bytes, stripes, k);
    else if (stripes) v = x_step(at_end, 0ull);

    // the quad's four accumulators to its first thread
    const uint32_t q0 = lane & ~3u;
    const unsigned long long v1 = __shfl_sync(0xFFFFFFFFu, v, q0), v2 = __shfl_sync(0xFFFFFFFFu, v, q0 + 1u),
                             v3 = __shfl_sync(0xFFFFFFFFu, v, q0 + 2u), v4 = __shfl_sync(0xFFFFFFFFu, v, q0 + 3u);
    if (k != 0u || row >= my_rows || c >= n_chunks) return;
    out[c] = x_finish(cache + (uint64_t)c * chunk_bytes, len, seed, v1, v2, v3, v4);
}

}  // namespace wm
