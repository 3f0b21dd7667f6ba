// wm_checksum: per-tile digests (k_tile_digests) and their fold into chunk CRCs (k_checksum_finish).
// Part of the one translation unit wm_kernels.cu (included there, in this order).
#pragma once

namespace wm {

// ------------------------------------------------------------------ wm_checksum

// Three kernels, by the size of the cache (the rule, with both sides' times, is checksum_any's).
//   k_chunk_crcs          small caches: a block takes one chunk and folds it itself; one launch
//   k_tile_digests        a team of eight warps per tile; k_checksum_finish folds the digests
//   k_tile_digests_stream large caches: a warp per tile; the same finish
// What bounds the last two is the shared memory the look-ups go through (128 bytes a cycle and SM):
// a tile is 512 look-ups of a warp in the chain, and with a team per tile 64 more at the ends of its
// eight warps' chains.

// The cleared control block: the error word in it is the call's outcome (wm_workspace_status).
__global__ void k_checksum_init(Ctrl* ctrl)
{
    grid_dep_wait();
    grid_dep_launch();
    if (threadIdx.x < sizeof(Ctrl) / 4) reinterpret_cast<uint32_t*>(ctrl)[threadIdx.x] = 0u;
}

// Small caches.  A block takes one chunk of at most TEAMS tiles, a tile per team, straight into
// registers, and thread 0 folds the chunk.  Nothing in
// here waits for a copy, so there is no outcome to report but success.
template <int TEAMS>
__global__ void __launch_bounds__(TEAMS * 256, 1)
k_chunk_crcs(const unsigned char* cache, Geo g, Ws ws, const Tables* __restrict__ tab, uint32_t* __restrict__ crc_out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wdig[TEAMS][8], s_rdig[8], s_dig[TEAMS];
    const uint32_t team = threadIdx.x / kTeamThreads, tt = threadIdx.x % kTeamThreads;
    const uint32_t warp = tt / 32, lane = tt % 32;
    const uint32_t c = blockIdx.x, t0 = c * g.tiles_per_chunk, t = t0 + team;
    const uint32_t ntc = min(g.tiles_per_chunk, g.n_tiles - t0);
    const bool full = team < ntc && t < g.n_full_tiles;
    const uint32_t ht = (&tab->HT[0][0])[threadIdx.x];
    Smem S = setup_smem(smem, tab);
    unsigned char* const slot = S.take(kTile);
    uint32_t* const sHT = reinterpret_cast<uint32_t*>(S.take(4096));        // (complete behind the block's barrier)
    sHT[threadIdx.x] = ht;
    grid_dep_wait();
    grid_dep_launch();
    if (c == 0 && threadIdx.x == 0) ws.ctrl->err = 0;
    uint32_t d[kWordsPerLane];
    if (full) {
        const uint32_t* p = reinterpret_cast<const uint32_t*>(cache + (uint64_t)t * kTile) + warp * 512u + lane;
#pragma unroll
        for (int i = 0; i < 16; i++) d[i] = __ldcs(p + 32 * i);
    }
    if (full) {
        const uint32_t v = tile_digest_part(S, d, team == 0u, warp, lane);
        if (lane == 0) s_wdig[team][warp] = v;
        team_bar(team);
        if (tt == 0) s_dig[team] = xor8(s_wdig[team]);
    } else if (team < ntc) {                   // the ragged last tile of the cache
        const uint32_t v = ragged_tile_digest(S, g, slot, cache + (uint64_t)t * kTile, s_rdig, team, tt);
        if (tt == 0) s_dig[team] = v;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const uint64_t clen = chunk_len_dev(g, c);
    if (clen < 4) {
        crc_out[c] = crc_bytewise(tab->T0, cache + (uint64_t)c * g.chunk_bytes, (uint32_t)clen);
        return;
    }
    uint32_t st = 0;
    for (uint32_t k = 0; k < ntc; k++)
        st = (t0 + k == g.n_full_tiles ? mulmod_dev(st, g.k_tail, g.poly) : advance_tile(sHT, st)) ^ s_dig[k];
    crc_out[c] = ~st;
}

struct DigTeamCtl {
    uint32_t wdig[2][8];
    unsigned long long mbar;
    unsigned long long pad;
};
static_assert(sizeof(DigTeamCtl) % 16 == 0, "team control block keeps 16-byte alignment");

// Tile digests, a team per tile: static striding over tiles.  Each team owns one 16 KiB stage that
// bulk copies (TMA) fill; the team takes its 16 words per lane out of the stage, hands the stage to
// the copy of its next tile and digests from registers meanwhile.
template <int TEAMS>
__global__ void __launch_bounds__(TEAMS * 256, 1)
k_tile_digests(const unsigned char* __restrict__ cache, Geo g, Ws ws, const Tables* __restrict__ tab)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Smem S = setup_smem(smem, tab);
    grid_dep_wait();
    grid_dep_launch();
    const uint32_t team = threadIdx.x / kTeamThreads, tt = threadIdx.x % kTeamThreads;
    const uint32_t warp = tt / 32, lane = tt % 32;
    unsigned char* stage = nullptr;
    for (int i = 0; i < TEAMS; i++) {          // every thread carves the same blocks in the same order
        unsigned char* p = S.take(kTile);
        if ((uint32_t)i == team) stage = p;
    }
    DigTeamCtl* tc = reinterpret_cast<DigTeamCtl*>(S.take(TEAMS * sizeof(DigTeamCtl)));
    if (!S.ok) { if (threadIdx.x == 0) atomicOr(&ws.ctrl->err, 4u); return; }
    tc += team;
    const uint64_t stride = (uint64_t)gridDim.x * TEAMS;
    const uint64_t pol = l2_policy_evict_first();
    auto start_copy = [&](uint64_t tile) {     // one thread of the team
        if (tile < g.n_full_tiles && !(g.inject & kInjectNoCopy)) bulk_load(stage, cache + tile * kTile, kTile, &tc->mbar, pol);
    };

    uint64_t t = (uint64_t)blockIdx.x * TEAMS + team;
    // the ragged last tile: by the team that comes by next in turn, before its loop
    if (g.tail_len && t == g.n_full_tiles % stride) {
        const uint32_t v = ragged_tile_digest(S, g, stage, cache + (uint64_t)g.n_full_tiles * kTile, tc->wdig[0], team, tt);
        if (tt == 0) ws.dig[g.n_full_tiles] = v;
        team_bar(team);
    }
    if (tt == 64u) { mbar_init(&tc->mbar, 1); start_copy(t); }
    team_bar(team);
    uint32_t phase = 0, par = 0;
    uint64_t t_done = ~0ull;                     // tile whose digest parts wait in wdig[par ^ 1]
    // One team barrier per tile.  The single-lane chores sit on different warps (the team waits
    // for whichever warp has the most to do): warp 2 starts the next copy, warp 1 folds and
    // stores the previous tile's digest once the barrier has made its parts complete.
    for (; t < g.n_full_tiles; t += stride) {
        const bool first = first_in_chunk(g, (uint32_t)t);
        uint32_t d[kWordsPerLane];
        wait_for_copy_at<false>((uint32_t)__cvta_generic_to_shared(&tc->mbar), phase, g.wait_ns, ws.ctrl, (g.inject & kInjectNoCopy) != 0u);
        phase ^= 1u;
        read_staged_words(stage, warp, lane, d);
        team_bar(team);                          // stage free; the previous tile's digest parts complete
        if (tt == 64u && phase < kStuck) start_copy(t + stride);
        if (tt == 32u && t_done != ~0ull) ws.dig[t_done] = xor8(tc->wdig[par ^ 1u]);
        const uint32_t v = tile_digest_part(S, d, first, warp, lane);
        if (lane == 0) tc->wdig[par][warp] = v;
        t_done = t;
        par ^= 1u;
    }
    team_bar(team);
    if (tt == 32u && t_done != ~0ull) ws.dig[t_done] = xor8(tc->wdig[par ^ 1u]);
}

// Tile digests, a warp per tile: its lanes' chains run over all 128 rows, so that a chain has one end
// per tile, no warp waits for another and there is nothing to put together.  A warp owns a 2 KiB stage
// that bulk copies fill, an eighth of a tile each; it takes 16 words per lane out of it, hands it to
// the next copy and walks on.  Tiles are dealt out warp by warp across the SMs, so that the SMs'
// shares differ by a tile at most.
__global__ void __launch_bounds__(1024, 1)
k_tile_digests_stream(const unsigned char* __restrict__ cache, Geo g, Ws ws, const Tables* __restrict__ tab)
{
    extern __shared__ __align__(16) unsigned char smem[];
    Smem S = setup_smem(smem, tab);
    grid_dep_wait();
    grid_dep_launch();
    const uint32_t warp = threadIdx.x / 32u, lane = threadIdx.x % 32u;
    unsigned char* const stages = S.take(32u * kShare);
    unsigned long long* const bars = reinterpret_cast<unsigned long long*>(S.take(32u * 8u));
    uint32_t* const wdig = reinterpret_cast<uint32_t*>(S.take(32u));
    if (!S.ok) { if (threadIdx.x == 0) atomicOr(&ws.ctrl->err, 4u); return; }
    // the ragged last tile: by the last team of the last block (one of those with the fewest tiles), whose stages make a tile's
    if (g.tail_len && blockIdx.x == gridDim.x - 1u && warp >= 24u) {
        const uint32_t tt = threadIdx.x - 768u;
        const uint32_t v = ragged_tile_digest(S, g, stages + 24u * kShare, cache + (uint64_t)g.n_full_tiles * kTile, wdig, 3, tt);
        if (tt == 0) ws.dig[g.n_full_tiles] = v;
    }
    const uint64_t pol = l2_policy_evict_first();
    const uint32_t stage_s = (uint32_t)__cvta_generic_to_shared(stages) + warp * kShare;
    const uint32_t bar_s = (uint32_t)__cvta_generic_to_shared(bars) + 8u * warp;
    const uint32_t stride = 32u * gridDim.x;
    uint32_t t = warp * gridDim.x + blockIdx.x;
    auto start_copy = [&](uint32_t tile, uint32_t part) {      // lane 0
        if (tile < g.n_full_tiles && !(g.inject & kInjectNoCopy))
            bulk_load_at(stage_s, cache + (uint64_t)tile * kTile + part * kShare, kShare, bar_s, pol);
    };
    if (lane == 0) { mbar_init(&bars[warp], 1); start_copy(t, 0); }
    __syncwarp();
    uint32_t phase = 0;
    for (; t < g.n_full_tiles; t += stride) {
        uint32_t s = first_in_chunk(g, t) && lane == 0u ? 0xFFFFFFFFu : 0u;      // (the all-ones start value complements the chunk's first word)
        for (uint32_t part = 0; part < 8u; part++) {
            wait_for_copy_at<true>(bar_s, phase, g.wait_ns, ws.ctrl, (g.inject & kInjectNoCopy) != 0u);
            phase ^= 1u;
            uint32_t w[kWordsPerLane];
            read_staged_words_at(stage_s, 0u, lane, w);
            __syncwarp();
            if (lane == 0 && phase < kStuck) start_copy(part < 7u ? t : t + stride, (part + 1u) & 7u);
            if (part) s = chain_step(S, s);
#pragma unroll
            for (int i = 0; i < 15; i++) s = chain_step(S, s ^ w[i]);
            s ^= w[15];
        }
        const uint32_t v = __reduce_xor_sync(0xFFFFFFFFu, lane_finish(S, s));
        if (lane == 0) ws.dig[t] = v;
    }
}

__global__ void __launch_bounds__(1024)
k_checksum_finish(const unsigned char* __restrict__ cache, Geo g, Ws ws, const Tables* __restrict__ tab,
                  uint32_t* __restrict__ crc_out)
{
    __shared__ uint32_t sHT[1024];
    __shared__ uint32_t sT0[256];
    __shared__ FinishStage stage;
    load_ht_t0(sHT, sT0, tab);
    grid_dep_wait();
    grid_dep_launch();
    const uint32_t c0 = blockIdx.x * g.finish_cb;
    stage_chunk_digests(g, stage, ws.dig, c0);
    const uint32_t c = c0 + threadIdx.x;
    // Fail closed: when the digest kernel reported trouble (a wait that ran out, no room for its
    // stages) some digests are not those of the cache.  The vector is then zero-filled and the
    // control block keeps the reason for wm_workspace_status.
    const bool failed = ld_volatile_u32(&ws.ctrl->err) != 0u;
    if (threadIdx.x < g.finish_cb && c < g.n_chunks)
        crc_out[c] = failed ? 0u : chunk_crc_staged(g, sHT, sT0, stage, ws.dig, cache + (uint64_t)c * g.chunk_bytes, c, threadIdx.x);
}

}  // namespace wm
