// Leaf mode: the table of tensors turned into one descriptor per tile (k_leaf_map), and the
// byte-exact readers / writers for the few tiles that do not sit inside one leaf.
// Part of the one translation unit wm_kernels.cu (included there, in this order).
#pragma once

namespace wm {

// ------------------------------------------------------------------ leaf tables

// The logical cache is the concatenation of `n` leaves (tensors) of any positive sizes; the
// 16 KiB tile grid is laid over that concatenation, so a tile may begin anywhere inside a leaf
// and may run across leaf boundaries (a scalar flag between two tensors, say).  k_leaf_map
// writes, per leaf, the logical offset at which it starts (ws.lstart, n + 1 entries) and, per
// tile, the address the main kernels use for it (ws.tptr):
//   - a tile whose 16384 bytes sit in one leaf, together with the 16-byte aligned block around
//     them: the address of its first byte inside the leaf.  It moves by a bulk copy from the
//     address rounded down to 16; the main kernels shift the words by the remainder.
//   - any other tile (it crosses a leaf boundary, or is the ragged last tile, or ends within 16
//     bytes of the end of a leaf whose size is no multiple of 16: the aligned block would reach
//     past the leaf) is a "walked" tile: it gets a 16 KiB slot in the workspace's side buffer and
//     its address is the slot's.  k_leaf_gather fills the slots from the leaves before the encode
//     kernel runs, k_leaf_scatter empties them into the leaves after the decode kernel has run,
//     both run by run, whole words inside a run, so the main kernels see ordinary aligned tiles and carry no
//     code for the exception.  There are at most two walked tiles per leaf; ws.wlist keeps their
//     numbers, ctrl->n_walked their count.
// Rules (a table that breaks one raises error bit 8; in decode mode it also closes the gate and
// writes the result record; nothing is read or written through a rejected table): 1..4096
// leaves, every pointer 16-byte aligned, every size positive and at most nbytes (so the sum
// cannot wrap), the sizes add up to nbytes, at most kMaxWalked walked tiles.

__global__ void __launch_bounds__(1024)
k_leaf_map(const wm_leaf* __restrict__ leaves, uint32_t n, Geo g, Ws ws, wm_result* result, int decode)
{
    __shared__ unsigned long long s_start[kMaxLeaves + 1];      // logical offset of each leaf; [n] = nbytes
    __shared__ unsigned long long s_wsum[32];
    __shared__ uint32_t s_bad;
    const uint32_t lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    grid_dep_wait();
    grid_dep_launch();
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    // thread i owns leaves 4i .. 4i+3
    unsigned long long len[4], mine = 0;
    uint32_t bad = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint32_t i = 4 * threadIdx.x + k;
        len[k] = 0;
        if (i < n) {
            const unsigned long long nb = leaves[i].nbytes;
            const unsigned long long p = reinterpret_cast<unsigned long long>(leaves[i].ptr);
            if (nb == 0 || nb > g.nbytes || p == 0 || (p & 15ull) != 0) bad = 1;
            len[k] = nb <= g.nbytes ? nb : 0;          // (a refused size must not wrap the sum)
            mine += len[k];
        }
    }
    unsigned long long incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned long long o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    if (lane == 31) s_wsum[warp] = incl;
    if (bad) s_bad = 1;
    __syncthreads();
    unsigned long long run = incl - mine;
    for (uint32_t w2 = 0; w2 < warp; w2++) run += s_wsum[w2];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint32_t i = 4 * threadIdx.x + k;
        if (i < n) s_start[i] = run;
        run += len[k];
    }
    if (threadIdx.x == 1023 && run != g.nbytes) s_bad = 1;      // the last thread's running sum is the total
    __syncthreads();
    if (threadIdx.x == 0) s_start[n] = g.nbytes;
    __syncthreads();
    auto refuse = [&]() {
        atomicOr(&ws.ctrl->err, 8u);
        if (decode) {
            ws.ctrl->gate = (uint32_t)WM_ERR_ARG;
            wm_result r;
            memset(&r, 0, sizeof r);
            r.status = WM_ERR_ARG;
            *result = r;
        }
    };
    if (s_bad) {
        if (blockIdx.x == 0 && threadIdx.x == 0) refuse();
        return;
    }
    if (blockIdx.x == 0)
        for (uint32_t i = threadIdx.x; i <= n; i += blockDim.x) ws.lstart[i] = s_start[i];
    const uint32_t n_slots = g.n_tiles < kMaxWalked ? g.n_tiles : kMaxWalked;
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < g.n_tiles; t += gridDim.x * blockDim.x) {
        const unsigned long long L0 = (unsigned long long)t * kTile;
        uint32_t lo = 0, hi = n;                       // the leaf with start[lo] <= L0 < start[lo + 1]
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) / 2;
            if (s_start[mid] <= L0) lo = mid; else hi = mid;
        }
        const unsigned long long in_leaf = L0 - s_start[lo];            // the tile's first byte inside its leaf
        const unsigned long long leaf_len = s_start[lo + 1] - s_start[lo];
        const unsigned long long addr = reinterpret_cast<unsigned long long>(leaves[lo].ptr) + in_leaf;
        const unsigned long long r = addr & 15ull;
        // whole, inside this leaf, and so is the aligned block that a shifted copy reads
        const bool direct = L0 + kTile <= g.nbytes && in_leaf + kTile + (r ? 16ull - r : 0ull) <= leaf_len;
        if (direct) {
            ws.tptr[t] = addr;
        } else {
            const uint32_t slot = atomicAdd(&ws.ctrl->n_walked, 1u);
            if (slot < n_slots) {
                ws.wlist[slot] = t;
                ws.tptr[t] = reinterpret_cast<unsigned long long>(ws.side + (size_t)slot * kTile);
            } else {
                ws.tptr[t] = 0ull;
                if (slot == n_slots) refuse();         // too many tiles cut by leaf boundaries for the side buffer
            }
        }
    }
}

// The runs of consecutive bytes a walked tile is made of (one per leaf it touches), handed to
// `f(leaf_bytes, tile_offset, run_length)`; every thread of the block goes through the same runs.
// The leaf a tile begins in is found by the whole block at once (a count of the leaves that start at
// or before it: one trip to L2, where a binary search is a dozen), and what the next 32 leaves are
// arrives in shared memory in one more.
struct RunStage {
    unsigned long long start[33];
    unsigned char* ptr[32];
};
template <typename F>
__device__ __forceinline__ void for_each_run(const wm_leaf* __restrict__ leaves, const unsigned long long* __restrict__ lstart,
                                             uint32_t n, const Geo& g, uint32_t t, RunStage& st, F f)
{
    const unsigned long long L0 = (unsigned long long)t * kTile;
    const uint32_t len = (uint32_t)min((unsigned long long)kTile, g.nbytes - L0);
    uint32_t before = 0;                                               // leaves that start at or before the tile (the first always does)
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < kMaxLeaves; i += 256u) {
        if (i - threadIdx.x >= n) break;
        before += (uint32_t)__syncthreads_count(i < n && __ldcg(lstart + i) <= L0);
    }
    uint32_t done = 0;
    for (uint32_t k0 = before - 1u; done < len && k0 < n; k0 += 32u) {
        __syncthreads();
        if (threadIdx.x < 33u && k0 + threadIdx.x <= n) st.start[threadIdx.x] = __ldcg(lstart + k0 + threadIdx.x);
        if (threadIdx.x < 32u && k0 + threadIdx.x < n)
            st.ptr[threadIdx.x] = const_cast<unsigned char*>(static_cast<const unsigned char*>(leaves[k0 + threadIdx.x].ptr));
        __syncthreads();
        for (uint32_t j = 0; j < 32u && done < len && k0 + j < n; j++) {
            const unsigned long long at = L0 + done;                   // first byte of the run (start[j] <= at < start[j + 1])
            const uint32_t run = (uint32_t)min((unsigned long long)(len - done), st.start[j + 1] - at);
            f(st.ptr[j] + (at - st.start[j]), done, run);
            done += run;
        }
    }
    __syncthreads();                                                   // the stage is free for the next tile
}

// A block copies `n` bytes between places of any alignment, reading nothing outside [src rounded
// down to 4, src + n) and writing nothing outside [dst, dst + n): whole words of the destination,
// each put together from two words of the source when the two are aligned differently, and a few
// bytes at either end.  The kernels below stand in front of the encode kernel and behind the decode
// kernel, so their time is exposed: with one byte per load and store they took 40 and 36 us for the
// 420 tiles of a table of 450 tensors; now 16 and 15.
__device__ __forceinline__ void copy_run(unsigned char* __restrict__ dst, const unsigned char* __restrict__ src, uint32_t n)
{
    const uint32_t head = min(n, (4u - ((uint32_t)reinterpret_cast<uintptr_t>(dst) & 3u)) & 3u);
    const uint32_t off = (uint32_t)reinterpret_cast<uintptr_t>(src + head) & 3u;
    // (a word put together from two reads up to three bytes past its own last one: the run's last word
    // is left to the byte loop)
    uint32_t words = (n - head) / 4u;
    if (off && words) words--;
    const uint32_t* p = reinterpret_cast<const uint32_t*>(src + head - off);
    uint32_t* q = reinterpret_cast<uint32_t*>(dst + head);
    // (a slot's 4096 words are at most 16 per thread: all of a thread's loads go out together)
    constexpr uint32_t kPer = kTile / 4u / 256u;
    uint32_t v[kPer];
#pragma unroll
    for (uint32_t k = 0; k < kPer; k++) {
        const uint32_t i = threadIdx.x + 256u * k;
        v[k] = 0u;
        if (i < words) v[k] = off == 0u ? __ldcg(p + i) : __funnelshift_r(__ldcg(p + i), __ldcg(p + i + 1), 8u * off);
    }
#pragma unroll
    for (uint32_t k = 0; k < kPer; k++) {
        const uint32_t i = threadIdx.x + 256u * k;
        if (i < words) q[i] = v[k];
    }
    const uint32_t rest = n - head - 4u * words;                       // at most 7
    if (threadIdx.x < head) dst[threadIdx.x] = __ldcg(src + threadIdx.x);
    if (threadIdx.x < rest) dst[n - rest + threadIdx.x] = __ldcg(src + n - rest + threadIdx.x);
}

// Encode: every walked tile copied from the leaves into its slot (one block per tile at a time).
__global__ void __launch_bounds__(256)
k_leaf_gather(const wm_leaf* __restrict__ leaves, uint32_t n, Geo g, Ws ws)
{
    grid_dep_wait();
    grid_dep_launch();
    if (ld_volatile_u32(&ws.ctrl->err) & 8u) return;
    __shared__ RunStage st;
    const uint32_t n_walked = ld_volatile_u32(&ws.ctrl->n_walked);
    for (uint32_t s = blockIdx.x; s < n_walked; s += gridDim.x) {
        unsigned char* slot = ws.side + (size_t)s * kTile;
        for_each_run(leaves, ws.lstart, n, g, ws.wlist[s], st, [&](const unsigned char* src, uint32_t off, uint32_t run) {
            copy_run(slot + off, src, run);
        });
    }
}

// Decode: every walked tile copied from its slot into the leaves.  Runs behind the decode kernel
// that stores; stays out when the gate is closed (nothing was decoded, the slots hold nothing).
__global__ void __launch_bounds__(256)
k_leaf_scatter(const wm_leaf* __restrict__ leaves, uint32_t n, Geo g, Ws ws)
{
    grid_dep_wait();
    grid_dep_launch();
    if (ld_volatile_u32(&ws.ctrl->gate)) return;
    __shared__ RunStage st;
    const uint32_t n_walked = ld_volatile_u32(&ws.ctrl->n_walked);
    for (uint32_t s = blockIdx.x; s < n_walked; s += gridDim.x) {
        const uint32_t t = ws.wlist[s];
        if (!(ld_volatile_u32(&ws.cflag[chunk_of(g, t)]) & CF_PRESENT)) continue;     // a tile of an absent chunk was not decoded
        const unsigned char* slot = ws.side + (size_t)s * kTile;
        for_each_run(leaves, ws.lstart, n, g, t, st, [&](unsigned char* dst, uint32_t off, uint32_t run) {
            copy_run(dst, slot + off, run);
        });
    }
}

}  // namespace wm
