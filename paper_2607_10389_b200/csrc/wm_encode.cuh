// wm_encode: placement (tickets, scanner warp), the single-pass fused checksum + encode kernel
// with its variants (mask, leaves, zero / constant tiles, entropy option), and its finish kernel.
// Part of the one translation unit wm_kernels.cu (included there, in this order).
#pragma once

namespace wm {

// ------------------------------------------------------------------ wm_encode

// Clears the control block and the placement words, zero-fills the padding behind the tile
// table.  With a dirty mask the main kernel claims the tiles of the present chunks only, so
// here the table entries of all tiles start at 0 (absent) and the first block lists the present
// chunks in ascending order (ws.plist; every thread a run of consecutive chunks, one prefix over
// the threads' counts) and leaves the number of tiles to claim in the control block.
__global__ void __launch_bounds__(1024)
k_encode_init(Geo g, Ws ws, unsigned char* wire, const uint8_t* dirty)
{
    grid_dep_wait();
    grid_dep_launch();
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = i; t < g.n_tiles; t += stride) ws.lbk[t] = 0u;
    if (i < sizeof(Ctrl) / 4) reinterpret_cast<uint32_t*>(ws.ctrl)[i] = 0u;
    // zero padding between the tile table and the payload
    const uint64_t tab_end = 64ull + 16ull * g.n_chunks + 2ull * g.n_tiles;
    if (i < g.meta_end - tab_end) wire[tab_end + i] = 0;
    __syncthreads();                                   // the control block is cleared before anything is written into it
    if (!dirty) {
        if (i == 0) ws.ctrl->n_tickets = g.n_tiles;
        return;
    }
    uint16_t* tile_tab = reinterpret_cast<uint16_t*>(wire + 64 + 16ull * g.n_chunks);
    for (uint64_t t = i; t < g.n_tiles; t += stride) tile_tab[t] = 0;
    if (blockIdx.x != 0) return;
    __shared__ uint32_t s_part[33];
    const uint32_t per = (g.n_chunks + 1023u) / 1024u;
    const uint32_t c0 = min(threadIdx.x * per, g.n_chunks), c1 = min(c0 + per, g.n_chunks);
    uint32_t mine = 0;
    for (uint32_t c = c0; c < c1; c++) mine += dirty[c] != 0 ? 1u : 0u;
    uint32_t n_listed;
    uint32_t at = block_prefix(mine, s_part, n_listed);
    for (uint32_t c = c0; c < c1; c++)
        if (dirty[c] != 0) ws.plist[at++] = c;
    if (threadIdx.x == 0) {
        // every present chunk has tiles_per_chunk tiles, except the cache's last chunk
        const uint32_t np = n_listed;
        uint32_t nt = np * g.tiles_per_chunk;
        if (np && dirty[g.n_chunks - 1]) nt -= g.tiles_per_chunk - (g.n_tiles - (g.n_chunks - 1) * g.tiles_per_chunk);
        ws.ctrl->n_list = np;
        ws.ctrl->n_tickets = nt;
    }
}

constexpr uint32_t kFlagA = 1u << 30, kFlagP = 2u << 30, kValMask = (1u << 30) - 1u;
constexpr uint32_t kUnit = 32;              // placement words count in units of 32 bytes

// Placement of the encoded tiles: a chained scan with one dedicated scanner warp.
//
// lbk[t] starts at 0.  The team that encodes tile t publishes kFlagA | len(t)/32 as soon as the
// length is known.  One scanner warp (alone in the block that wins a lock at kernel start, so
// that it has an SM's issue slots to itself) walks the array in order, 256 entries per poll,
// turns every leading run of published lengths into kFlagP | (exclusive prefix)/32, and moves
// on.  The owner of tile t then reads its offset back from lbk[t].  Every encoded length that
// another tile has to add is a multiple of 32 (only the cache's last tile can be ragged, and
// nothing follows it); 30 bits of 32-byte units cover 32 GiB of payload.
//
// Several hundred tiles are in flight at any time and publish at about the same moment;
// letting each of them walk back to the nearest finished prefix made the walk, not the data,
// the bottleneck, and assigning tiles statically made every round wait for its slowest team.
// The scanner is running by construction (it won the lock), tiles are claimed in ticket
// order, and a team publishes the length of a claimed tile without waiting for anyone, so the
// owners' waits depend only on running code; they are bounded all the same, by time (the call's
// wait budget), and end in WM_ERR_TIMEOUT.
__device__ __forceinline__ void st_relaxed_u32(uint32_t* p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t next_ticket(Ctrl* ctrl)
{
    return atomicAdd(&ctrl->ticket, 1u);
}

// Owner side: exclusive prefix (bytes) of tile t (one lane spins, for at most `budget_ns`; the
// poison flag and the clock are looked at every 64 polls).
__device__ __forceinline__ unsigned long long wait_prefix(const uint32_t* lbk, uint32_t t, Ctrl* ctrl, uint32_t budget_ns)
{
    const uint32_t t0 = now_ns();
    for (uint32_t polls = 0;; polls++) {
        const uint32_t v = ld_relaxed_u32(lbk + t);
        if ((v >> 30) == 2u) return (unsigned long long)(v & kValMask) * kUnit;
        if ((polls & 63u) == 63u && (ld_volatile_u32(&ctrl->poison) || now_ns() - t0 > budget_ns)) break;
    }
    give_up(ctrl);
    return 0;
}

// Scanner side (one full warp).  A poll fetches 256 consecutive entries, lane l four of either half in
// one 16-byte load (one round trip to L2), and turns the leading run of published ones into offsets.
// The time of a poll is what every owner's offset waits for, so nothing in it is spread out: a half's
// entries lie across the lanes as they lie in memory, both ways one coalesced access, and the two
// halves' prefix sums run side by side.  (512 entries through shared memory, sixteen consecutive ones
// per lane with a store each, took 1.5 us a poll, this takes 1.0.)
__device__ __forceinline__ uint4 ld_now_v4(const uint32_t* p)
{
    uint4 v;
    asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ void scan_tile_lengths(uint32_t* lbk, uint32_t n_tiles, uint32_t lane, Ctrl* ctrl, uint32_t budget_ns)
{
    uint32_t f = 0;                 // first unresolved entry
    uint32_t base = 0;              // units before f
    uint32_t spins = 0;             // polls in a row that resolved nothing
    uint32_t t0 = 0;                // the clock when that run of empty polls began
    while (f < n_tiles) {
        const uint32_t w0 = f & ~3u;                      // 16-byte aligned window start
        uint32_t v[2][4], cnt[2], sum[2], incl[2], lead[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t at = w0 + 128u * h + 4u * lane;                   // (the entries are padded to a multiple of 4)
            const uint4 x = at < n_tiles ? ld_now_v4(lbk + at) : make_uint4(0u, 0u, 0u, 0u);
            v[h][0] = x.x; v[h][1] = x.y; v[h][2] = x.z; v[h][3] = x.w;
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            // the lane's leading published entries (those before f are done: they count, with value 0)
            const uint32_t at = w0 + 128u * h + 4u * lane;
            cnt[h] = 0; sum[h] = 0;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const bool done = at + j < f;
                if (cnt[h] == (uint32_t)j && at + j < n_tiles && (done || (v[h][j] >> 30) == 1u)) {
                    cnt[h]++;
                    sum[h] += done ? 0u : v[h][j] & kValMask;
                }
            }
            const uint32_t fm = __ballot_sync(0xFFFFFFFFu, cnt[h] == 4u);
            lead[h] = fm == 0xFFFFFFFFu ? 32u : (uint32_t)(__ffs(~fm) - 1);      // leading full lanes
        }
        if (lead[0] < 32u) lead[1] = 0xFFFFFFFFu;          // the run ends in the first half: nothing of the second counts
#pragma unroll
        for (int h = 0; h < 2; h++) {
            if (lead[h] == 0xFFFFFFFFu || lane > lead[h]) { cnt[h] = 0; sum[h] = 0; }
            incl[h] = sum[h];
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl[h], d);
                if (lane >= (uint32_t)d) incl[h] += o;
            }
        }
        const uint32_t all0 = __shfl_sync(0xFFFFFFFFu, incl[0], 31), all1 = __shfl_sync(0xFFFFFFFFu, incl[1], 31);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t at = w0 + 128u * h + 4u * lane;
            const uint32_t r0 = base + (h ? all0 : 0u) + incl[h] - sum[h];       // units before the lane's first new entry
            if (cnt[h] == 4u && at >= f) {
                const uint32_t r1 = r0 + (v[h][0] & kValMask), r2 = r1 + (v[h][1] & kValMask), r3 = r2 + (v[h][2] & kValMask);
                asm volatile("st.volatile.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(lbk + at), "r"(kFlagP | r0), "r"(kFlagP | r1), "r"(kFlagP | r2),
                             "r"(kFlagP | r3) : "memory");
            } else {
                uint32_t run = r0;
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    if ((uint32_t)j < cnt[h] && at + j >= f) {
                        st_relaxed_u32(lbk + at + j, kFlagP | run);
                        run += v[h][j] & kValMask;
                    }
                }
            }
        }
        const uint32_t k_all = __reduce_add_sync(0xFFFFFFFFu, cnt[0] + cnt[1]);  // entries from w0 on that are resolved now
        const uint32_t k = w0 + k_all - f;
        base += all0 + all1;
        f += k;
        if (k == 0) {
            // nothing new: the owners are behind.  Every 64 such polls in a row the scanner looks at the
            // poison flag and at the clock; it gives up when no length has come in for the whole budget.
            if (spins == 0u) t0 = now_ns();
            if ((++spins & 63u) == 0u) {
                const bool stop = ld_volatile_u32(&ctrl->poison) != 0u || now_ns() - t0 > budget_ns;
                if (__any_sync(0xFFFFFFFFu, stop)) {
                    if (lane == 0) give_up(ctrl);
                    return;
                }
            }
        } else {
            spins = 0;
        }
    }
}

__device__ __forceinline__ uint32_t desc_of(uint32_t base, uint32_t w)
{
    return base | (w << 8) | ((((base & 15u) ^ (base >> 4) ^ w ^ 5u) & 15u) << 12);
}

// A team of the encode kernel: four warps.  Warp w owns rows 32w .. 32w+31 of the tile, that is shares
// (16 rows, four groups) 2w and 2w + 1, one after the other.
constexpr uint32_t kEncTeams = 8, kEncTeamThreads = 128;
struct EncTeamCtl {
    uint32_t wtab[4][32];   // per group: base | w << 8 (| marks on a share's first entry), by step modulo 4
    uint32_t wdig[4][4];    // per warp: its block's digest
    uint32_t etab[4][8];    // entropy option, per share: anchor | words of its stream << 8 (0xFFFF: a strand too long for the form)
    uint32_t ssum[4];       // sum of the 32 widths of the tile (set by the publishing warp), or a mark:
                            // zero tile, constant tile, kSumEnt | words of the streams for a tile stored in ENT form
    uint32_t next[2];       // the tile to be measured two steps after it was put here, by step parity
    uint32_t pad[2];
    uint32_t kring[8];      // with a mask: the ticket of a tile in flight, by step modulo 8 (placement runs over tickets)
    unsigned long long excl[2];   // offset of the tile packed in the next step, by step parity
    unsigned long long nptr[2];   // leaf mode: address (k_leaf_map) of the tile in next[], by step parity
    unsigned long long mbar[4];   // per warp: completion of the bulk copy into its stage
    unsigned long long measured;  // the four warps' measures of the step's tile are complete
    unsigned long long pad2;
    unsigned char sbits[2][256];  // entropy option: every strand's bit length - 64, by step parity (a warp reads its
                                  // own strands only, before it writes the next ones)
};
static_assert(sizeof(EncTeamCtl) % 16 == 0, "team control block keeps 16-byte alignment");
__device__ __forceinline__ void enc_team_bar(uint32_t team)
{
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(kEncTeamThreads) : "memory");
}

__device__ __forceinline__ void stg_u8(void* p, uint32_t v)
{
    asm volatile("st.global.cs.u8 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void stg_u16(void* p, uint32_t v)
{
    asm volatile("st.global.cs.u16 [%0], %1;" ::"l"(p), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void stg_v2(void* p, uint32_t a, uint32_t b)
{
    asm volatile("st.global.cs.v2.u32 [%0], {%1, %2};" ::"l"(p), "r"(a), "r"(b) : "memory");
}

// Write the bit planes of one group straight to the wire image.  The lane holds the eight
// exponent bytes of its elements (e4a, e4b, coded order); after the base is subtracted each
// is < 2^W.  W = 8 is stored as it is; otherwise a 4-bit, a 2-bit and a 1-bit plane (those
// whose bit is set in W) take consecutive bits of the deltas from bit 0.  In every plane lane
// l owns an aligned 4 / 2 / 1-byte unit at l times that size, so each warp store covers one
// contiguous, sector-aligned run of 128 / 64 / 32 bytes and nothing needs staging.
//   nibbles : the low nibbles of v and the high ones of v >> 4 put two 4-bit values side by side in
//             bytes 0 and 2 of each word (bits above the plane fall away)
//   2 bits  : (t * 0x01041040) >> 24 gathers the four 2-bit fields of a word into one byte
//   1 bit   : (t * 0x01020408) >> 24 gathers the four bits of a word into one nibble
// (the partial products of both multiplications land on distinct bits, so no carry occurs).
// Width 4 is by far the most frequent; the others share one piece of code that goes plane by plane
// (seven pieces, four times each in the loop, were more than the instruction cache wants to hold).
__device__ __forceinline__ void pack_nibbles(uint32_t da, uint32_t db, unsigned char* p, uint32_t lane)
{
    const uint32_t va = (da & 0x0F0F0F0Fu) | ((da >> 4) & 0xF0F0F0F0u), vb = (db & 0x0F0F0F0Fu) | ((db >> 4) & 0xF0F0F0F0u);
    st_stream_u32(p + 4 * lane, __byte_perm(va, vb, 0x6420));
}
__device__ __forceinline__ void pack_group(uint32_t wd, uint32_t e4a, uint32_t e4b, uint32_t base, unsigned char* p, uint32_t lane)
{
    const uint32_t b4 = base * 0x01010101u;
    uint32_t da = e4a - b4, db = e4b - b4;
    if (wd == 4u) {
        pack_nibbles(da, db, p, lane);
    } else if (wd == 8u) {
        stg_v2(p + 8 * lane, da, db);
    } else {
        if (wd & 4u) {
            pack_nibbles(da, db, p, lane);
            p += 128;
            da >>= 4; db >>= 4;
        }
        if (wd & 2u) {
            const uint32_t pa = (da & 0x03030303u) * 0x01041040u, pb = (db & 0x03030303u) * 0x01041040u;
            stg_u16(p + 2 * lane, __byte_perm(pa, pb, 0x0073));
            p += 64;
            da >>= 2; db >>= 2;
        }
        if (wd & 1u) {
            const uint32_t pa = (da & 0x01010101u) * 0x01020408u, pb = (db & 0x01010101u) * 0x01020408u;
            const uint32_t x = __byte_perm(pa, pb, 0x0073);          // byte 0: a's nibble, byte 1: b's nibble
            stg_u8(p + lane, x | (x >> 4));
        }
    }
}


// ---- ENT tiles: entropy-coded exponents (an encoder option; header flags bit 2) --------------
// A warp's 2 KiB of a tile (16 rows) is one share; lane l's 32 elements (its 16 words, low half
// first) are strand l.  Every exponent is coded as u = E - anchor with a fixed prefix code, the
// anchor being the rounded mean of the share's exponents; a strand is the LSB-first bit string of
// its 32 codewords, and the 32 strands of a share lie one behind the other in the share's
// stream, their lengths written down in a byte each, so that every lane of the reading warp
// finds the start of its strand with one prefix sum and nobody waits for anybody.
//   u        -6  -5  -4  -3  -2  -1   0   1   2   3   other
//   length    8   6   5   4   4   2   2   2   4   7   16 (eight ones, then E itself)
//   bits    127  31  15  11   3   2   0   1   7  63   255 | E << 8        (first bit = bit 0)
// ent_slot: 0..9 for u = -6..3, 10 for everything else.
__device__ __forceinline__ uint32_t ent_slot(uint32_t E, uint32_t anchor)
{
    return min(E - anchor + 6u, 10u);
}
// Both tables are byte look-ups done with permutes (no branches: the lanes of a warp hold
// different slots): slots 0..7 from one pair of words, 8..10 from a third.
__device__ __forceinline__ uint32_t ent_lut(uint32_t lo, uint32_t hi, uint32_t top, uint32_t slot)
{
    const uint32_t a = __byte_perm(lo, hi, slot), b = __byte_perm(top, 0u, slot & 7u);
    return (slot < 8u ? a : b) & 0xFFu;
}
__device__ __forceinline__ uint32_t ent_length(uint32_t slot)
{
    return ent_lut(0x04050608u, 0x02020204u, 0x00100704u, slot);      // 8 6 5 4 | 4 2 2 2 | 4 7 16
}
__device__ __forceinline__ uint32_t ent_word(uint32_t slot, uint32_t E)
{
    const uint32_t w = ent_lut(0x0B0F1F7Fu, 0x01000203u, 0x00FF3F07u, slot);       // 127 31 15 11 | 3 2 0 1 | 7 63 255
    return w | (slot == 10u ? E << 8 : 0u);
}
// Bytes of an ENT tile whose eight streams hold `words` 32-bit words in all (a multiple of 32;
// 16384 or more means that the tile takes another form): header, sign-mantissa plane, strand
// lengths, streams.
__device__ __forceinline__ uint32_t ent_tile_bytes(uint32_t words)
{
    return (8512u + 4u * words + 31u) & ~31u;
}
// Decoder side.  A codeword is s ones and a zero (s < 8; eight ones: the escape), followed for
// s = 0 and s = 2 by one more bit x:  s = 0: u = -x;  1: +1;  2: -2 - x;  3: +2;  4..7: -4, -5, +3, -6.
// ent_ones: s, capped at 8, of the codeword at the low end of `buf` (zero beyond the valid bits).
__device__ __forceinline__ uint32_t ent_ones(uint32_t buf)
{
    return min((uint32_t)__ffs(~buf) - 1u, 8u);
}
__device__ __forceinline__ uint32_t ent_parse_length(uint32_t s)
{
    const uint32_t l = __byte_perm(0x04040202u, 0x08070605u, s & 7u) & 0xFFu;       // 2 2 4 4 | 5 6 7 8
    return s == 8u ? 16u : l;
}
__device__ __forceinline__ uint32_t ent_parse_value(uint32_t buf, uint32_t s, uint32_t anchor)
{
    const uint32_t base = __byte_perm(0x02FE0100u, 0xFA03FBFCu, s & 7u);            // 0 +1 -2 +2 | -4 -5 +3 -6
    const uint32_t x = ((s & 5u) == 0u) ? (buf >> (s + 1u)) & 1u : 0u;
    return s == 8u ? (buf >> 8) & 0xFFu : (anchor + base - x) & 0xFFu;
}

// Single-pass fused checksum + encode.  Each team keeps three tiles in flight:
//     X  measured two steps ago, packed and written to the wire image in this step
//     W  measured in the last step, at the end of which its length was published
//     Y  checksummed and measured in this step
// Every warp has a 2 KiB stage of its own in shared memory that bulk copies (TMA) fill, a share (16
// rows) at a time; it takes 16 words per lane out of it and starts the next copy at once, so a warp
// waits for its own data and the team meets at one barrier per tile.  A measured share's words are
// parked in tensor memory (four shares per warp: two tiles) until the tile's offset is known, so a
// tile is read from memory once and nothing waits in registers.  Per step:
//     team barrier | fetch X's two shares and pack them straight into the wire image | take Y's two
//     shares: digest, exponent ranges, park | publish len(Y)
// The chores of a step sit on different warps: the team passes one barrier per tile, so it runs at the
// pace of the warp that has the most to do.
// What bounds it is the number of instructions issued, then the time an offset takes to come back.
// Teams of eight warps with one share each and one stage per team met twice as often and did the
// step's bookkeeping once per share: 11 % more instructions, 596 us on the engine cache (1.67 GB)
// against 526 us, 449 -> 412 with a mask, 604 -> 565 in leaf mode, 1178 -> 1123 with the entropy option.
// The four shares per warp that tensor memory holds leave one step between a length and its offset;
// with lengths published behind the next team barrier, and tickets claimed a step earlier, late
// offsets held back the lengths that other offsets waited for, and the kernel fell to 767 us.
// Template switches: MASKED (a dirty mask was given), LEAVES (the cache is a table of tensors), ZEROS (the zero / constant tile option), ENT (the entropy option: the measuring step also
// adds up codeword lengths, the tile takes the shorter of the two coded forms, and for the ENT
// form the packing step writes the strands' lengths and the share's stream of words instead of bit planes).
// Packed data goes from registers to the wire image directly: in every region of a PACK tile
// a lane owns an aligned unit at a lane-strided place, so each warp store is one contiguous
// sector-aligned run.  Claiming a tile before the previous offset is known means that, if the
// scanner is late, this team waits while that tile's length is not out yet; with a whole step
// of slack that is rare, and it only delays: the teams that hold earlier tiles never depend
// on this one.
// A tile as a team passes it round: its number in the low 22 bits, kQFirst when it is the first
// tile of its chunk; the top bit alone (kQNone): no tile.  Leaf mode adds, in bits 22-25, how many
// bytes above a 16-byte boundary the tile starts.  (The codec takes caches of at most 2^21 tiles.)
// Only full tiles are passed round: the ragged last tile is the scanner's block's business.
constexpr uint32_t kQNone = 1u << 31, kQFirst = 1u << 30, kQTile = (1u << 22) - 1u;
constexpr uint32_t kQOffShift = 22;
// Marks in a team's width table: on a share's first entry, all 2 KiB of its rows are zero;
// as the sum of the widths, the tile is all zero.
// kWarpConst: all 1024 elements of the share's rows hold one value (its sign-mantissa byte rides in
// bits 16-23 of the entry, the exponent is the base); kSumConstTile: the tile holds one value.
constexpr uint32_t kWarpAllZero = 0x8000u, kWarpConst = 0x4000u, kSumZeroTile = 0xFFFFu, kSumConstTile = 0xFFFEu;
constexpr uint32_t kSumRaw = 256u;          // as the sum of the widths: stored raw (any sum above 253 is)
// The tile is stored in ENT form (shorter than its bit planes and than raw); low half: words of its streams.
constexpr uint32_t kSumEnt = 0x10000u;

// The tile behind ticket k.  Without a mask tickets are tile numbers.  With one, only the tiles of
// present chunks are claimed: ticket k is tile k mod tiles_per_chunk of the (k / tiles_per_chunk)-th
// present chunk (plist, ascending, written by k_encode_init), so placement runs over tickets and a
// sparse mask costs nothing for what it leaves out.  n_hot: tickets of full tiles.
template <bool MASKED>
__device__ __forceinline__ uint32_t describe_tile(const Geo& g, const uint32_t* plist, uint32_t n_hot, uint32_t k)
{
    if (k >= n_hot) return kQNone;
    uint32_t t = k;
    bool first = first_in_chunk(g, k);
    if (MASKED) {
        const uint32_t j = chunk_of(g, k);
        t = __ldcg(plist + j) * g.tiles_per_chunk + (k - j * g.tiles_per_chunk);
    }
    return t | (first ? kQFirst : 0u);
}

// The ragged last tile (ticket k, behind all others), stored raw: by the second team of the scanner's
// block, beside the scanner.  Nothing follows it, so its length is of no interest to the scanner: the
// zero published here only asks for the tile's offset.
__device__ __forceinline__ void encode_ragged_tile(const Smem& S, const Geo& g, const unsigned char* __restrict__ tile, unsigned char* __restrict__ wire,
                                                uint64_t wire_cap, const Ws& ws, uint32_t k, unsigned char* slot, uint32_t* wdig)
{
    const uint32_t tt = threadIdx.x % kTeamThreads, t = g.n_full_tiles;
    __shared__ unsigned long long s_excl;
    if (tt == 0) st_relaxed_u32(ws.lbk + k, kFlagA);
    const uint32_t v = ragged_tile_digest(S, g, slot, tile, wdig, 1, tt);
    if (tt == 0) {
        ws.dig[t] = v;
        s_excl = wait_prefix(ws.lbk, k, ws.ctrl, g.wait_ns);
    }
    team_bar(1);
    const unsigned long long excl = s_excl;
    if (tt == 0) {
        reinterpret_cast<uint16_t*>(wire + 64 + 16ull * g.n_chunks)[t] = 0xFFFFu;
        if (first_in_chunk(g, t)) *reinterpret_cast<unsigned long long*>(wire + 64 + 16ull * chunk_of(g, t)) = excl;
        ws.ctrl->payload_total = excl + g.tail_len;
        if (excl + g.tail_len > wire_cap - g.meta_end) atomicOr(&ws.ctrl->err, 1u);
    }
    if (excl + g.tail_len <= wire_cap - g.meta_end) copy_ragged_tile(wire + g.meta_end + excl, tile, g.tail_len, tt);
}

template <bool MASKED, bool LEAVES, bool ZEROS, bool ENT = false>
__global__ void __launch_bounds__(kEncTeams * kEncTeamThreads, 1)
k_encode(const unsigned char* __restrict__ cache, Geo g, const uint8_t* __restrict__ dirty,
         unsigned char* __restrict__ wire, uint64_t wire_cap, Ws ws, const Tables* __restrict__ tab)
{
    extern __shared__ __align__(16) unsigned char smem[];
    // The first block to get here becomes the scanner: one warp of it, alone on its SM (a warp
    // that shares its scheduler with busy ones gets too few issue slots to keep up).
    __shared__ uint32_t s_scanner;
    __shared__ uint32_t s_tmem;
    Smem S = setup_smem(smem, tab);
    grid_dep_wait();                   // from here on the control block and the length table are ready
    grid_dep_launch();
    if (LEAVES && (ld_volatile_u32(&ws.ctrl->err) & 8u)) return;      // the leaf table was rejected
    if (threadIdx.x == 0) s_scanner = atomicCAS(&ws.ctrl->scan_lock, 0u, 1u) == 0u;
    __syncthreads();
    // Tickets: all of them, and those of full tiles (the teams').  The ragged last tile of the cache,
    // when its chunk is present, is the last ticket.
    const uint32_t n_tickets = MASKED ? ld_volatile_u32(&ws.ctrl->n_tickets) : g.n_tiles;
    const bool ragged = g.tail_len != 0u && (!MASKED || dirty[g.n_chunks - 1u] != 0);
    const uint32_t n_hot = ragged ? n_tickets - 1u : n_tickets;
    if (s_scanner) {
        unsigned char* slot = S.take(kTile);
        uint32_t* wdig = reinterpret_cast<uint32_t*>(S.take(32));
        if (!S.ok) { if (threadIdx.x == 0) atomicOr(&ws.ctrl->err, 4u); return; }
        // (test hook: with the scanner left out no offset is ever handed out, and the owners' waits run out)
        if (threadIdx.x < 32 && !(g.inject & kInjectNoScanner)) scan_tile_lengths(ws.lbk, n_tickets, threadIdx.x, ws.ctrl, g.wait_ns);
        if (ragged && threadIdx.x / kTeamThreads == 1u)
            encode_ragged_tile(S, g, LEAVES ? reinterpret_cast<const unsigned char*>(ws.tptr[g.n_full_tiles]) : cache + (uint64_t)g.n_full_tiles * kTile,
                               wire, wire_cap, ws, n_tickets - 1u, slot, wdig);
        return;
    }
    const uint32_t team = threadIdx.x / kEncTeamThreads, tt = threadIdx.x % kEncTeamThreads;
    const uint32_t wc = threadIdx.x / 32, warp = tt / 32, lane = tt % 32;
    // (leaf mode: a tile may start off a 16-byte boundary; a copy then starts at the boundary
    // below and is 16 bytes longer, so the stage is too)
    constexpr uint32_t kStage = LEAVES ? kShare + 16u : kShare;
    unsigned char* const stages = S.take(kEncTeams * 4u * kStage);
    EncTeamCtl* tc = reinterpret_cast<EncTeamCtl*>(S.take(kEncTeams * sizeof(EncTeamCtl)));
    // ENT: codeword length and codeword by k = E - anchor + 256 (1..511), so that a look-up is the
    // exponent added to an address the share works out once (no slot arithmetic per element); the
    // escape's codeword reads 0xFFFF (the packing step lets the exponent through its high byte)
    unsigned char* const t_lenE = ENT ? S.take(512) : nullptr;
    unsigned short* const t_cwE = ENT ? reinterpret_cast<unsigned short*>(S.take(1024)) : nullptr;
    if (!S.ok) { if (threadIdx.x == 0) atomicOr(&ws.ctrl->err, 4u); return; }
    tc += team;
    if (ENT && threadIdx.x < 512u) {
        const int u = (int)threadIdx.x - 256;
        const uint32_t slot = (u >= -6 && u <= 3) ? (uint32_t)(u + 6) : 10u;
        t_lenE[threadIdx.x] = (unsigned char)ent_length(slot);
        t_cwE[threadIdx.x] = (unsigned short)(slot == 10u ? 0xFFFFu : ent_word(slot, 0u));
    }
    const uint32_t lenE_s = ENT ? (uint32_t)__cvta_generic_to_shared(t_lenE) + 256u : 0u;
    const uint32_t cwE_s = ENT ? (uint32_t)__cvta_generic_to_shared(t_cwE) + 512u : 0u;

    // Tensor memory for the tiles in flight: allocated by the block's first warp, the address
    // goes round through shared memory.  Warp w of the block owns lanes 32 (w % 4) .. + 31 and
    // 64 columns from 64 (w / 4): four slots of 16 columns, two shares of two tiles.
    if (threadIdx.x < 32) tmem_alloc_all(&s_tmem);
    tmem_fence_before_sync();
    __syncthreads();
    tmem_fence_after_sync();
    const uint32_t tmem_warp = s_tmem + ((32u * (wc & 3u)) << 16) + 64u * (wc >> 2);

    unsigned char* const payload = wire + g.meta_end;
    const uint64_t room = wire_cap - g.meta_end;                 // payload bytes that fit
    const uint64_t pol_once = l2_policy_evict_first();           // every tile is read once
    const uint32_t stage_s = (uint32_t)__cvta_generic_to_shared(stages) + wc * kStage;
    const uint32_t tc_s = (uint32_t)__cvta_generic_to_shared(tc);
    const uint32_t bar_s = tc_s + (uint32_t)offsetof(EncTeamCtl, mbar) + 8u * warp;
    const bool leader = (tt == 0);
    uint32_t stuck = 0;                // kStuck when a copy into the stage has not come
    uint32_t measured_phase = 0;       // warp 3: parity of the measures', kStuck when a wait for them has run out

    auto is_tile = [](uint32_t q) { return (int32_t)q >= 0; };
    // (the placement words are indexed by ticket: with a mask that is the tile's entry in kring, else the tile number)
    auto place_of = [&](uint32_t step, uint32_t q) { return MASKED ? tc->kring[step & 7u] : q & kQTile; };
    // where tile t lives: its address in the flat cache, or (leaf mode) the address that k_leaf_map wrote
    auto tile_src = [&](uint32_t t) -> unsigned long long {
        return LEAVES ? ws.tptr[t] : reinterpret_cast<unsigned long long>(cache + (uint64_t)t * kTile);
    };
    // Lane 0 of a warp, when the warp's stage is free (never again once it is stuck): the copy of one of its two shares.  Leaf mode: a
    // tile may start off a 16-byte boundary; the copy then starts at the boundary below and takes 16
    // bytes more (k_leaf_map saw to it that they belong to the leaf); the readers shift by the remainder.
    auto start_copy = [&](uint32_t q, unsigned long long src, uint32_t part) {
        if (!is_tile(q | stuck)) return;
        const unsigned long long a = (LEAVES ? src & ~15ull : src) + kShare * (2u * warp + part);
        bulk_load_at(stage_s, reinterpret_cast<const void*>(a), (LEAVES && (src & 15ull)) ? kShare + 16u : kShare, bar_s, pol_once);
    };
    // leaf mode, handing a claimed tile on: its word carries the start's remainder
    auto with_mark = [](uint32_t q, unsigned long long addr) {
        return (!LEAVES || (int32_t)q < 0) ? q : q | (((uint32_t)addr & 15u) << kQOffShift);
    };

    // Tiles in flight, oldest first: X (packed in this step), W (its length goes out), Y (measured in
    // this step).  Y's results go to the tables' slot step mod 4 and to tensor memory slot step mod 2.
    uint32_t qX = kQNone, qW = kQNone, qY = kQNone;
    uint32_t step = 0;
    bool claiming = false;             // leader: the last ticket it claimed was a tile

    // ---- prologue: the tiles of the first two steps are claimed.  Up to a tile per team, a block runs as
    // many teams as it takes to share the tiles out evenly, and a team draws one ticket at first.  Up to
    // two per team, as many teams of every block as its share asks for have a second tile; it comes behind
    // all teams' first ones in ticket order, and nobody draws any more.  (First come, first served, the
    // second tiles all went to the blocks that had started first, and those ran twice as long as the
    // others: 24 MB 36.0 us, 24 MB with the entropy option 51.3, now 29.9 and 42.6.)  With more tiles than
    // that a team draws two at first and goes on from there.
    if (leader) {
        const uint32_t per_block = (n_hot + gridDim.x - 2u) / (gridDim.x - 1u);
        const bool one = per_block <= kEncTeams, many = per_block > 2u * kEncTeams;
        uint32_t k0 = 0xFFFFFFFFu, k1 = 0xFFFFFFFFu;
        if (team < per_block) k0 = next_ticket(ws.ctrl);
        if (many && k0 < n_hot) k1 = next_ticket(ws.ctrl);        // (behind the answer: the teams' second tiles come after most first ones)
        else if (team + kEncTeams < per_block) k1 = kEncTeams * (gridDim.x - 1u) + atomicAdd(&ws.ctrl->second, 1u);
        const uint32_t q0 = describe_tile<MASKED>(g, ws.plist, n_hot, k0);
        const uint32_t q1 = describe_tile<MASKED>(g, ws.plist, n_hot, k1);
        // (with a tile per team at most the next draw finds nothing, but it keeps the teams from their offsets
        // until the scanner has them: without it 8 to 17 MB took 0.9 us longer, measured on four forms of this.
        // Not with the entropy option, whose draws come too early for that and where it takes nothing.)
        claiming = is_tile(many ? q1 : q0) && (many || (one && !ENT));
        if (MASKED) { tc->kring[0] = k0; tc->kring[1] = k1; }      // the steps in which they will be measured
        tc->next[0] = q0;
        tc->next[1] = q1;
        tc->excl[0] = 0ull;
        tc->excl[1] = 0ull;
        if (LEAVES) {
            tc->nptr[0] = is_tile(q0) ? tile_src(q0 & kQTile) : 0ull;
            tc->nptr[1] = is_tile(q1) ? tile_src(q1 & kQTile) : 0ull;
            tc->next[0] = with_mark(q0, tc->nptr[0]);
            tc->next[1] = with_mark(q1, tc->nptr[1]);
        }
    }
    if (lane == 0) mbar_init(&tc->mbar[warp], 1);
    if (tt == 96u) mbar_init(&tc->measured, (g.inject & kInjectNoMeasures) ? 5 : 4);      // (test hook: the fifth never comes)
    enc_team_bar(team);
    qY = tc->next[0];
    unsigned long long srcY = LEAVES ? tc->nptr[0] : 0ull;      // leaf mode: where Y begins
    if (lane == 0) start_copy(qY, LEAVES ? srcY : tile_src(qY & kQTile), 0);

    uint32_t trouble = 0;              // sticky: the image does not fit
    uint32_t d[kWordsPerLane];
    while (is_tile(qX & qW & qY)) {
        enc_team_bar(team);            // W's widths and digests are complete; what was handed over in the last step is visible
        const uint32_t par = step & 1u;
        const uint32_t slX = (step - 2u) & 3u, slW = (step - 1u) & 3u, slY = step & 3u;
        const uint32_t qN = tc->next[par ^ 1u];
        const unsigned long long exclX = tc->excl[par ^ 1u];
        const unsigned long long srcN = LEAVES ? tc->nptr[par ^ 1u] : 0ull;

        // ---- W: warp 1 puts its digest together
        if (warp == 1u && is_tile(qW)) {
            const uint32_t v = place_team4_digests(S, tc_s + (uint32_t)offsetof(EncTeamCtl, wdig) + 16u * slW, lane);
            if (lane == 0) ws.dig[qW & kQTile] = v;
        }
        // Round trips to L2 are under way during a step whose answers are taken at its end: W's offset (asked
        // for by warp 2 in front of Y's second share) and the ticket of the tile to measure two steps on
        // (the leader).  Without mask, leaves and entropy option it is claimed as late as that allows, in the
        // middle of the step: the time from a claim to the tile's length, times how unevenly the teams
        // run, is what an offset waits for.  With a mask or leaves a ticket is looked up once more (its
        // chunk's number, its address): it is claimed at the start of the step and looked up in the middle.
        // With the entropy option it is claimed at the start as well: where tiles of very different lengths
        // follow one another, teams that claim late stand at their offsets (a text model's window of
        // 1.61 GB, three quarters zeros, 967 us late and 832 early, with zero tiles 1368 and 788, Gaussian
        // and random pieces in turn 1318 and 892; attention caches 1076 and 1080).
        constexpr bool kEarly = MASKED || LEAVES || ENT;
        uint32_t pv = 0, tk = 0xFFFFFFFFu, qC = kQNone, plA = 0;
        unsigned long long pA = 0;
        if (kEarly && leader && claiming) tk = next_ticket(ws.ctrl);
        auto ask = [&]() {
            if (tt == 64u && is_tile(qW)) pv = ld_relaxed_u32(ws.lbk + place_of(step - 1u, qW));
            if (leader && claiming) {
                if (!kEarly) {
                    tk = next_ticket(ws.ctrl);
                } else if ((MASKED || LEAVES) && tk < n_hot) {
                    if (LEAVES) { qC = describe_tile<MASKED>(g, ws.plist, n_hot, tk); pA = tile_src(qC & kQTile); }
                    else plA = __ldcg(ws.plist + chunk_of(g, tk));
                }
            }
        };

        // ---- X: its words back from tensor memory, packed straight into the wire image
        if (is_tile(qX)) {
            const uint32_t Smark = tc->ssum[slX];
            const bool ent_form = ENT && (Smark & kSumEnt) != 0u;
            const uint32_t Ssum = ent_form ? Smark & 0xFFFFu : Smark;       // words of the streams, or the sum of the widths
            const bool packs = !ent_form && Ssum <= 253u;
            // (a tile of all-zero bytes, marked in ssum, is its table entry and nothing else)
            const uint32_t enc_len = ent_form ? ent_tile_bytes(Ssum)
                                         : packs ? 8256u + 32u * Ssum : (ZEROS && Ssum == kSumZeroTile) ? 0u
                                         : (ZEROS && Ssum == kSumConstTile) ? 32u : kTile;
            unsigned char* const dst = payload + exclX;
            tmem_wait_stores();
            if (exclX + enc_len > room) {
                trouble |= 1u;
            } else if (ent_form) {
                // header: anchors, word counts, 40 zero bytes; zero fill behind the last stream
                if (warp == 2u) {
                    if (lane < 8u) {
                        const uint32_t wt = tc->etab[slX][lane];
                        stg_u8(dst + lane, wt & 0xFFu);
                        stg_u16(dst + 8u + 2u * lane, wt >> 8);
                    } else if (lane < 18u) {
                        st_stream_u32(dst + 24u + 4u * (lane - 8u), 0u);
                    }
                    if (4u * lane < enc_len - 8512u - 4u * Ssum) st_stream_u32(dst + 8512u + 4u * Ssum + 4u * lane, 0u);
                }
#pragma unroll 1
                for (uint32_t part = 0; part < 2u; part++) {
                    const uint32_t share = 2u * warp + part;
                    tmem_load16(tmem_warp + 32u * par + 16u * part, d);
                    unsigned char* const sm_dst = dst + 64u + 1024u * share + 8u * lane;
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const uint32_t sa = __byte_perm(d[4 * j], d[4 * j + 1], 0x6420), sb = __byte_perm(d[4 * j + 2], d[4 * j + 3], 0x6420);
                        const uint32_t ya = __byte_perm(sa, sa, 0x2301), yb = __byte_perm(sb, sb, 0x2301);
                        stg_v2(sm_dst + 256 * j, (sa & 0xFEFEFEFEu) | (ya & 0x01010101u), (sb & 0xFEFEFEFEu) | (yb & 0x01010101u));
                    }
                    // This share's stream starts behind the streams of the shares before it; inside it the
                    // strands follow one another bit by bit, so lane l starts where the lengths of the
                    // lanes before it (measured two steps ago) add up to.
                    const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, lane < share ? tc->etab[slX][lane] >> 8 : 0u);
                    const uint32_t anchor = tc->etab[slX][share] & 0xFFu;
                    const uint32_t nb8 = tc->sbits[par][32u * share + lane];
                    stg_u8(dst + 8256u + 32u * share + lane, nb8);
                    uint32_t incl = 64u + nb8;
#pragma unroll
                    for (int k = 1; k < 32; k <<= 1) {
                        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, k);
                        if (lane >= (uint32_t)k) incl += o;
                    }
                    const uint32_t start = incl - 64u - nb8;
                    unsigned char* const w_dst = dst + 8512u + 4u * before;
                    // acc: the stream's bits from the last word boundary on, n of them valid (the first n
                    // of the lane's first word belong to the lane before it).  Two codewords are joined
                    // first (32 bits at most) and go in together; both shifts are multiplications by a
                    // power of two from the table or from n (one multiply-add each, on the pipe that has
                    // little else to do here, where the shifts and ORs would queue up with everything
                    // else).  Words go out as they fill up, except the lane's first one, which is held
                    // back until the lane before has handed over the bits it left in it.
                    unsigned long long acc = 0;
                    uint32_t n = start & 31u, wp = start >> 5, w_first = 0;
                    bool have_first = false;
                    const uint32_t lb = lenE_s - anchor, cb = cwE_s - 2u * anchor;
#pragma unroll
                    for (int i = 0; i < 16; i++) {
                        const uint32_t len0 = lds_tab_u8(__dp4a(d[i], 0x00000100u, lb)), len1 = lds_tab_u8(__dp4a(d[i], 0x01000000u, lb));
                        // (the table's escape entry is 0xFFFF: the AND lets the exponent, which is in the
                        // second byte of the word or of its high half, through there only)
                        const uint32_t c0 = lds_tab_u16(__dp4a(d[i], 0x00000200u, cb)) & (d[i] | 0xFFFF00FFu);
                        const uint32_t c1 = lds_tab_u16(__dp4a(d[i], 0x02000000u, cb)) & ((d[i] >> 16) | 0xFFFF00FFu);
                        const uint32_t pair = c1 * (1u << len0) + c0;
                        asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc) : "r"(pair), "r"(1u << n));
                        n += len0 + len1;
                        if (n >= 32u) {                        // (two codewords are 32 bits at most: one word per pair)
                            const uint32_t word = (uint32_t)acc;
                            if (have_first) st_stream_u32(w_dst + 4u * wp, word); else w_first = word;
                            have_first = true;
                            acc >>= 32;
                            n -= 32u;
                            wp++;
                        }
                    }
                    // (a strand is 64 bits at least, so every lane has crossed a word boundary by now)
                    const uint32_t tail = (uint32_t)acc;                   // n bits of the next word, 0 when n == 0
                    const uint32_t from_below = __shfl_up_sync(0xFFFFFFFFu, tail, 1);
                    st_stream_u32(w_dst + 4u * (start >> 5), w_first | (lane ? from_below : 0u));
                    if (lane == 31u && n) st_stream_u32(w_dst + 4u * wp, tail);
                }
            } else if (packs) {
                if (warp == 2u) {
                    const uint32_t wt = tc->wtab[slX][lane];
                    stg_u16(dst + 2 * lane, desc_of(wt & 0xFFu, (wt >> 8) & 15u));
                }
                // widths of all 32 groups (one per lane): 32-byte units before this warp's first group
                const uint32_t wall = (tc->wtab[slX][lane] >> 8) & 15u;
                unsigned char* rec = dst + 8256u + 32u * __reduce_add_sync(0xFFFFFFFFu, lane < 8u * warp ? wall : 0u);
                unsigned char* sm_dst = dst + 64u + 2048u * warp + 8u * lane;      // this lane's place in a group's sign-mantissa run
#pragma unroll 1
                for (uint32_t part = 0; part < 2u; part++) {
                    tmem_load16(tmem_warp + 32u * par + 16u * part, d);
                    const uint4 g4 = *reinterpret_cast<const uint4*>(&tc->wtab[slX][8u * warp + 4u * part]);
                    const uint32_t gq[4] = {g4.x, g4.y, g4.z, g4.w};
                    auto groups = [&](auto all4) {
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const uint32_t wtg = gq[j];
                        const uint32_t base = wtg & 0xFFu, wd = (wtg >> 8) & 15u;
                        // bytes 0 and 2 of a rotated word: mantissa << 1 | the other element's sign;
                        // bytes 1 and 3: the exponents.  Gather, then swap bit 0 inside byte pairs.
                        const uint32_t sa = __byte_perm(d[4 * j], d[4 * j + 1], 0x6420), sb = __byte_perm(d[4 * j + 2], d[4 * j + 3], 0x6420);
                        const uint32_t ya = __byte_perm(sa, sa, 0x2301), yb = __byte_perm(sb, sb, 0x2301);
                        stg_v2(sm_dst + 256 * j, (sa & 0xFEFEFEFEu) | (ya & 0x01010101u), (sb & 0xFEFEFEFEu) | (yb & 0x01010101u));
                        const uint32_t e4a = __byte_perm(d[4 * j], d[4 * j + 1], 0x7531), e4b = __byte_perm(d[4 * j + 2], d[4 * j + 3], 0x7531);
                        if (decltype(all4)::value) {
                            const uint32_t b4 = base * 0x01010101u;
                            pack_nibbles(e4a - b4, e4b - b4, rec + 128 * j, lane);
                        } else {
                            pack_group(wd, e4a, e4b, base, rec, lane);
                            rec += 32u * wd;
                        }
                    }
                    };
                    // (four groups of width 4, what most shares are: the planes' places are fixed)
                    if ((((g4.x ^ 0x400u) | (g4.y ^ 0x400u) | (g4.z ^ 0x400u) | (g4.w ^ 0x400u)) & 0xF00u) == 0u) {
                        groups(std::true_type());
                        rec += 512;
                    } else {
                        groups(std::false_type());
                    }
                    sm_dst += 1024;
                }
            } else if (ZEROS && Ssum == kSumConstTile) {
                // the value (any word's low half, rotated back), then 30 zero bytes
                tmem_load16(tmem_warp + 32u * par, d);
                if (warp == 2u && lane < 8u) st_stream_u32(dst + 4u * lane, lane == 0u ? __funnelshift_r(d[0], d[0], 1) & 0xFFFFu : 0u);
            } else if (enc_len) {
#pragma unroll 1
                for (uint32_t part = 0; part < 2u; part++) {
                    tmem_load16(tmem_warp + 32u * par + 16u * part, d);
                    unsigned char* q = dst + (2u * warp + part) * kShare + lane * 4u;
#pragma unroll
                    for (int i = 0; i < 16; i++) st_stream_u32(q + i * 128, __funnelshift_r(d[i], d[i], 1));
                }
            }
        }
        // What is left to note about X: the table entry, where its chunk starts, the total.
        if (tt == 32u && is_tile(qX)) {
            const uint32_t tXn = qX & kQTile, Ssum = tc->ssum[slX];
            uint32_t entry, enc_len;
            if (ENT && (Ssum & kSumEnt)) {
                enc_len = ent_tile_bytes(Ssum & 0xFFFFu);
                entry = 0x8000u | (enc_len / 32u);
            } else {
                entry = Ssum <= 253u ? 258u + Ssum : (ZEROS && Ssum == kSumZeroTile) ? 1u : (ZEROS && Ssum == kSumConstTile) ? 2u : 512u;
                enc_len = (ZEROS && entry <= 2u) ? 32u * (entry - 1u) : 32u * entry;
            }
            reinterpret_cast<uint16_t*>(wire + 64 + 16ull * g.n_chunks)[tXn] = (uint16_t)entry;
            if (qX & kQFirst) *reinterpret_cast<unsigned long long*>(wire + 64 + 16ull * chunk_of(g, tXn)) = exclX;
            if (place_of(step - 2u, qX) + 1 == n_tickets) ws.ctrl->payload_total = exclX + enc_len;
        }
        // ---- Y: digest, exponent ranges, words parked, a share at a time
        if (is_tile(qY)) {
            // Warp 3 adds up the 32 widths and publishes the tile's length: in the middle of its second share's
            // digest when the other warps' widths are there by then, else at the end of its own measuring,
            // not behind the next team barrier: that one waits for W's offset, and an offset that comes late
            // must not hold back a length that other teams' offsets are waiting for.
            // When the wait for the widths runs out (the call has failed then) nothing in the tables can be
            // trusted, now or in any later step: the tile and all that follow it are published as raw, whose
            // length is the same whatever the widths turn out to be, so that the packing step, which checks
            // the published length against the room in the wire buffer, never writes more than that.
            bool published = false;
            auto publish = [&](bool complete) {
                measured_phase ^= 1u;
                published = true;
                const uint32_t wt = tc->wtab[slY][lane];
                const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, (wt >> 8) & 15u), total = complete ? sum : kSumRaw;
                // entropy option: the ENT form is taken when it is shorter than the planes and than raw
                uint32_t ent_words = 0;
                if (ENT) ent_words = __reduce_add_sync(0xFFFFFFFFu, lane < 8u ? tc->etab[slY][lane] >> 8 : 0u);
                const uint32_t plane_len = total <= 253u ? 8256u + 32u * total : kTile;
                const bool ent_tile = ENT && complete && ent_tile_bytes(ent_words) < plane_len;
                // unused memory (every share's first entry carries the mark): no payload
                // (one value throughout: every share's first entry carries the mark and they are all alike;
                // a tile of zeros has no payload, any other value 32 bytes)
                const uint32_t wt0 = __shfl_sync(0xFFFFFFFFu, wt, 0);
                const bool const_tile = ZEROS && complete && __all_sync(0xFFFFFFFFu, (lane & 3u) != 0u || ((wt & kWarpConst) != 0u && wt == wt0));
                const bool zero_tile = const_tile && (wt0 & kWarpAllZero) != 0u;
                if (lane == 0) {
                    tc->ssum[slY] = zero_tile ? kSumZeroTile : const_tile ? kSumConstTile : ent_tile ? kSumEnt | ent_words : total;
                    const uint32_t len = zero_tile ? 0u : const_tile ? 32u : ent_tile ? ent_tile_bytes(ent_words) : plane_len;
                    st_relaxed_u32(ws.lbk + place_of(step, qY), kFlagA | (len / kUnit));
                }
            };
            uint32_t st = ((qY & kQFirst) && tt == 0u) ? 0xFFFFFFFFu : 0u;      // (the all-ones start value complements the chunk's first word)
            // (both shares written out: the second one's wait, loads and first look-ups come up beside the first
            // one's measuring; 518 -> 510 us, masked 399 -> 394, leaf mode 549 -> 541.  The packing loop above is
            // better left a loop: 513 when it is unrolled too.)
#pragma unroll
            for (uint32_t part = 0; part < 2u; part++) {
                const uint32_t share = 2u * warp + part;
                uint32_t phase = part | stuck;        // (two copies a tile: the first one's phase is even)
                wait_for_copy_at<true>(bar_s, phase, g.wait_ns, ws.ctrl);
                stuck = phase & kStuck;
                // leaf mode: a tile that was copied from the 16-byte boundary below it starts that many
                // bytes into the stage: whole words from a quarter of that on, each put together from two
                // neighbours when the remainder is no multiple of four
                const uint32_t off = LEAVES ? (qY >> kQOffShift) & 15u : 0u;
                const uint32_t sh = (off & 3u) * 8u;
                if (LEAVES && sh) {
                    const uint32_t* const p = reinterpret_cast<const uint32_t*>(stages + wc * kStage + (off & 12u)) + lane;
#pragma unroll
                    for (int i = 0; i < 16; i++) d[i] = __funnelshift_r(p[i * 32], p[i * 32 + 1], sh);
                } else {
                    read_staged_words_at(stage_s + (off & 12u), 0u, lane, d);
                }
                __syncwarp();
                if (lane == 0) {
                    if (part == 0u) start_copy(qY, LEAVES ? srcY : tile_src(qY & kQTile), 1u);
                    else start_copy(qN, LEAVES ? srcN : tile_src(qN & kQTile), 0u);
                }
                auto chain = [&](int from, int to) {
#pragma unroll
                    for (int i = from; i < to; i++) st = i < 15 ? chain_step(S, st ^ d[i]) : st ^ d[i];
                };
                // The words are kept rotated left by one bit: each half then reads [E | mantissa | a sign bit],
                // E in its high byte (the two sign bits of a word land in each other's half; the packing
                // step puts them right).
                auto rotate = [&]() {
#pragma unroll
                    for (int i = 0; i < 16; i++) d[i] = __funnelshift_l(d[i], d[i], 1);
                };
                // The second share's widths come before its digest, off the words with their signs cleared
                // (one instruction a word more): the sooner a length is out, the less an offset is waited
                // for.  With incompressible data, where a step is short, that wait was 30 % of a step and
                // the engine cache's size took 640 us; now 533 to 547.  An 8 MB cache's call: 20.5 -> 17.4 us.
                // (The last of the four warps publishing at once, found by a counter: 538 us, but 520 instead
                // of 508 on the engine cache, as the slowest warp then has the most to do; the first share's
                // widths moved forward as well: 528.  With the entropy option the measuring needs the
                // rotated words all the same and a step is long: digest first.)
                const bool early = !ENT && part != 0u;
                if (part) {
                    if (ENT) ask();
                    st = chain_step(S, st);
                }
                if (!early) {
                    chain(0, 16);
                    rotate();
                }
                auto word = [&](int i) { return early ? d[i] & 0x7FFF7FFFu : d[i]; };
                const uint32_t exp_shift = early ? 23u : 24u;
                uint32_t gw[4];               // per group: base | width << 8
                uint32_t ent_w = 0;           // entropy option: anchor | words << 8 of this share
                if (ENT) {
                    // the share's anchor (rounded mean of its 1024 exponents: bytes 1 and 3 of a rotated
                    // word), every strand's length in bits and the words the share's stream needs
                    uint32_t acc = 0;
#pragma unroll
                    for (int i = 0; i < 16; i++) acc = __dp4a(d[i], 0x01000100u, acc);       // bytes 1 and 3
                    const uint32_t anchor = (__reduce_add_sync(0xFFFFFFFFu, acc) + 512u) >> 10;
                    // (the exponents are bytes 1 and 3 of a rotated word: the dot product that picks one
                    // and adds the table's address is the look-up's whole address arithmetic)
                    uint32_t bits = 0;
                    const uint32_t lb = lenE_s - anchor;
#pragma unroll
                    for (int i = 0; i < 16; i++)
                        bits += lds_tab_u8(__dp4a(d[i], 0x00000100u, lb)) + lds_tab_u8(__dp4a(d[i], 0x01000000u, lb));
                    // (a strand the length byte cannot hold, above 319 bits, keeps the tile out of the form:
                    // the count is then so large that the form is never the shortest)
                    const uint32_t share_bits = __reduce_add_sync(0xFFFFFFFFu, bits);
                    const bool too_long = __any_sync(0xFFFFFFFFu, bits > 319u);
                    tc->sbits[par][32u * share + lane] = (unsigned char)(bits - 64u);
                    ent_w = anchor | ((too_long ? 0xFFFFu : (share_bits + 31u) >> 5) << 8);
                }
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const uint32_t a0 = word(4 * j), a1 = word(4 * j + 1), a2 = word(4 * j + 2), a3 = word(4 * j + 3);
                    uint32_t mn = min_u16x2(min_u16x2(a0, a1), min_u16x2(a2, a3));
                    uint32_t mx = max_u16x2(max_u16x2(a0, a1), max_u16x2(a2, a3));
                    // both halves get the smaller (larger) of the two, so that the word as a whole
                    // orders like its halves and one warp reduction per bound does
                    mn = min_u16x2(mn, __byte_perm(mn, mn, 0x1032));
                    mx = max_u16x2(mx, __byte_perm(mx, mx, 0x1032));
                    const uint32_t emin = __reduce_min_sync(0xFFFFFFFFu, mn) >> exp_shift;
                    const uint32_t emax = __reduce_max_sync(0xFFFFFFFFu, mx) >> exp_shift;
                    gw[j] = emin | ((32u - __clz(emax - emin)) << 8);
                }
                // Option ZEROS.  Unused memory: when all four groups have exponent 0 throughout (rare in live data)
                // look at the words themselves; a share whose 2 KiB are all zero marks its first entry.
                // The same for any one value (a mask fill, say): all four groups have one exponent and width
                // 0; then every word must equal the share's first, and that word's two halves each other.
                if (ZEROS && gw[0] < 256u && gw[1] == gw[0] && gw[2] == gw[0] && gw[3] == gw[0]) {
                    const uint32_t first = __shfl_sync(0xFFFFFFFFu, d[0], 0);
                    uint32_t diff = (first >> 16) ^ (first & 0xFFFFu);
#pragma unroll
                    for (int i = 0; i < 16; i++) diff |= d[i] ^ first;
                    if (!__any_sync(0xFFFFFFFFu, diff != 0u))
                        gw[0] |= kWarpConst | (((early ? first << 1 | first >> 31 : first) & 0xFFu) << 16) | (first == 0u ? kWarpAllZero : 0u);
                }
                if (lane == 0) {
                    *reinterpret_cast<uint4*>(&tc->wtab[slY][4u * share]) = make_uint4(gw[0], gw[1], gw[2], gw[3]);
                    if (ENT) tc->etab[slY][share] = ent_w;
                }
                if (part && lane == 0) mbar_arrive_at(tc_s + (uint32_t)offsetof(EncTeamCtl, measured));
                if (early) {
                    ask();                       // (here, not in front of the widths: 586 -> 550 us with incompressible data)
                    chain(0, 8);
                    if (warp == 3u && measured_phase < kStuck &&
                        __all_sync(0xFFFFFFFFu, mbar_test(tc_s + (uint32_t)offsetof(EncTeamCtl, measured), measured_phase)))
                        publish(true);
                    chain(8, 16);
                    rotate();
                }
                tmem_store16(tmem_warp + 32u * par + 16u * part, d);
            }
            const uint32_t v = __reduce_xor_sync(0xFFFFFFFFu, lane_finish(S, st));
            if (lane == 0) tc->wdig[slY][warp] = v;
            if (warp == 3u && !published) {
                wait_for_copy_at<true>(tc_s + (uint32_t)offsetof(EncTeamCtl, measured), measured_phase, g.wait_ns, ws.ctrl, true);
                if (__any_sync(0xFFFFFFFFu, measured_phase >= kStuck)) measured_phase |= kStuck;
                publish(measured_phase < kStuck);
            }
        } else {
            if (lane == 0) start_copy(qN, LEAVES ? srcN : tile_src(qN & kQTile), 0u);
            ask();
        }

        // ---- hand over: the tile to measure two steps on, and W's offset
        if (leader) {
            uint32_t qn = kQNone;
            if (tk < n_hot) {
                if (LEAVES) {
                    qn = with_mark(qC, pA);
                    tc->nptr[par] = pA;
                } else if (MASKED) {
                    const uint32_t j = chunk_of(g, tk);
                    qn = (plA * g.tiles_per_chunk + (tk - j * g.tiles_per_chunk)) | (first_in_chunk(g, tk) ? kQFirst : 0u);
                } else {
                    qn = describe_tile<false>(g, ws.plist, n_hot, tk);
                }
            }
            claiming = claiming && is_tile(qn);
            tc->next[par] = qn;
            if (MASKED) tc->kring[(step + 2u) & 7u] = tk;
        }
        if (tt == 64u) {
            unsigned long long e = 0;
            if (is_tile(qW))
                e = (pv >> 30) == 2u ? (unsigned long long)(pv & kValMask) * kUnit : wait_prefix(ws.lbk, place_of(step - 1u, qW), ws.ctrl, g.wait_ns);
            tc->excl[par] = e;
        }
        qX = qW; qW = qY; qY = qN;
        srcY = srcN;
        step++;
    }
    if ((trouble & 1u) && lane == 0) atomicOr(&ws.ctrl->err, 1u);
    // every warp is done with its tensor memory: hand it back before the block exits
    tmem_wait_stores();
    tmem_fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) tmem_free_all(s_tmem);
}

// Chunk c's directory entry and CRC (the calling thread's chunk: c0 + i).  Returns its term of the
// whole-cache CRC; `present` says whether the image carries it.
__device__ __forceinline__ uint32_t close_chunk(const unsigned char* __restrict__ cache, const Geo& g, const uint8_t* __restrict__ dirty,
                                                uint32_t* __restrict__ crc_inout, unsigned char* wire, const Ws& ws, const uint32_t* sHT,
                                                const uint32_t* sT0, const FinishStage& stage, const ChunkPowers& cp, unsigned long long total,
                                                uint32_t c, uint32_t i, uint32_t& present)
{
    unsigned char* dir = wire + 64;
    present = (!dirty || dirty[c]) ? 1u : 0u;
    // Where the chunk's payload starts: a present chunk's offset was written by the team that
    // placed its first tile; an absent chunk (the main kernel never saw it) starts where the next
    // present chunk does, or at the end of the payload.
    const uint32_t n_list = dirty ? ld_volatile_u32(&ws.ctrl->n_list) : 0u;
    auto starts_at = [&](uint32_t cc) -> unsigned long long {
        if (cc >= g.n_chunks) return total;
        if (!dirty || dirty[cc]) return *reinterpret_cast<const unsigned long long*>(dir + 16ull * cc);
        uint32_t lo = 0, hi = n_list;              // the first listed chunk above cc
        while (lo < hi) {
            const uint32_t mid = (lo + hi) / 2;
            if (ws.plist[mid] < cc) lo = mid + 1; else hi = mid;
        }
        return lo < n_list ? *reinterpret_cast<const unsigned long long*>(dir + 16ull * ws.plist[lo]) : total;
    };
    const unsigned long long po = starts_at(c), nx = starts_at(c + 1);
    uint32_t crc;
    if (present) {
        crc = chunk_crc_staged(g, sHT, sT0, stage, ws.dig, chunk_first_byte(g, ws, cache, c), c, i);
        crc_inout[c] = crc;
    } else {
        crc = crc_inout[c];
        *reinterpret_cast<unsigned long long*>(dir + 16ull * c) = po;
    }
    *reinterpret_cast<uint32_t*>(dir + 16ull * c + 8) = (uint32_t)(nx - po);
    *reinterpret_cast<uint32_t*>(dir + 16ull * c + 12) = crc;
    return cache_crc_term(g, cp, crc, c);
}

// The header (one thread; meta_crc left zero).
__device__ __forceinline__ void write_header(const Geo& g, unsigned char* wire, bool masked, uint32_t option_flags, uint32_t n_present,
                                             unsigned long long total, uint32_t cache_crc)
{
    uint32_t* h = reinterpret_cast<uint32_t*>(wire);
    h[0] = 0x31564D57u;                                  // "WMV1"
    h[1] = 1u | ((masked ? 1u : 0u) << 16) | (option_flags << 16);      // version, flags (bit 1 zero tiles, bit 2 ENT tiles)
    h[2] = (uint32_t)g.nbytes; h[3] = (uint32_t)(g.nbytes >> 32);
    h[4] = g.chunk_bytes; h[5] = kTile; h[6] = g.n_chunks; h[7] = n_present;
    h[8] = (uint32_t)total; h[9] = (uint32_t)(total >> 32);
    const unsigned long long wl = g.meta_end + total;
    h[10] = (uint32_t)wl; h[11] = (uint32_t)(wl >> 32);
    h[12] = cache_crc; h[13] = 0u; h[14] = 0u; h[15] = 0u;
}

// Directory (enc_len, crc), chunk CRCs, present count; the last block to finish combines the
// chunk CRCs into the cache CRC and writes the header (meta_crc left zero).
__global__ void __launch_bounds__(1024)
k_encode_finish(const unsigned char* __restrict__ cache, Geo g, const uint8_t* __restrict__ dirty,
                uint32_t* __restrict__ crc_inout, unsigned char* __restrict__ wire, Ws ws,
                const Tables* __restrict__ tab, const __grid_constant__ ChunkPowers cp, uint32_t option_flags)
{
    __shared__ uint32_t sHT[1024];
    __shared__ uint32_t sT0[256];
    __shared__ FinishStage stage;
    __shared__ uint32_t s_acc;
    __shared__ bool s_last;
    load_ht_t0(sHT, sT0, tab);
    grid_dep_wait();
    grid_dep_launch();
    const uint32_t c0 = blockIdx.x * g.finish_cb;
    stage_chunk_digests(g, stage, ws.dig, c0);
    const unsigned long long total = ws.ctrl->payload_total;
    // only finish_cb threads of a block fold chunks (the lookups of a full block would queue up
    // on one SM's shared memory)
    const uint32_t c = c0 + threadIdx.x;
    uint32_t present = 0, term = 0;
    const bool dead = (ld_volatile_u32(&ws.ctrl->err) & 8u) != 0;      // leaf mode: the table was rejected
    if (!dead && threadIdx.x < g.finish_cb && c < g.n_chunks)
        term = close_chunk(cache, g, dirty, crc_inout, wire, ws, sHT, sT0, stage, cp, total, c, threadIdx.x, present);
    accumulate_cache_crc(ws.ctrl, term, &s_acc);
    const uint32_t cnt = __syncthreads_count(present);
    if (threadIdx.x == 0) {
        if (cnt) atomicAdd(&ws.ctrl->n_present, cnt);
        __threadfence();
        s_last = atomicAdd(&ws.ctrl->done_a, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last || threadIdx.x != 0) return;
    __threadfence();
    const uint32_t cache_crc = ld_volatile_u32(&ws.ctrl->cache_acc);
    const uint32_t n_present = ld_volatile_u32(&ws.ctrl->n_present);
    write_header(g, wire, dirty != nullptr, option_flags, n_present, total, cache_crc);
    ws.ctrl->hdr_cache_crc = cache_crc;
    ws.ctrl->hdr_n_present = n_present;
    ws.ctrl->payload_total = total;
}

}  // namespace wm
