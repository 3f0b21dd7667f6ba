// The decode kernel's loop for large images: a warp per tile.  (wm_decode.cuh has the other one, a
// team of eight warps per tile, and decides.)
// Part of the one translation unit wm_kernels.cu (included there, in this order).
#pragma once

namespace wm {

// A warp's stage: one share of a tile.  PACK: 1 KiB of sign-mantissa bytes, then at most 1 KiB of planes.
// Raw: 2 KiB.  ENT: sign-mantissa bytes, 32 strand lengths, the share's stream from the 16-byte boundary
// below it on (12 + 4 * 319 + 28 bytes at most: the last share's runs to the tile's end).
constexpr uint32_t kDecStage = 2368, kDecPlanes = 1024, kDecStream = 1056;
// A warp's control block: its barrier, where its next tile's payload begins, where that tile goes, and 64
// bytes for answers about it (its header in the end).  Not in registers: there are none to spare.
constexpr uint32_t kDecCtl = 96, kDecSrc = 8, kDecDst = 16, kDecBuf = 32;

// A warp owns a tile and walks through its eight shares.  Nothing in here waits for another warp: no team
// barrier, one end of the checksum chain and one look at the header per tile instead of per share, the
// groups' places by a running sum.  A share is a copy (or two, or three) of its own into the warp's stage,
// started as soon as the share before has been taken out of it.  During a tile its successor is
// prepared, one dependent step per share: ticket (share 0), with a mask the chunk (1), table entry and
// offsets (2 to 4), header (4 to 6), first copy (7).
// DECODE_STREAM_FIGURES
template <bool LEAVES, int MODE, int ENT>
__device__ __forceinline__ void decode_stream(Smem& S, const unsigned char* __restrict__ wire, const Geo& g, unsigned char* __restrict__ dst, const Ws& ws,
                                              bool masked, uint32_t n_tickets, uint32_t ptab_s)
{
    __shared__ uint32_t s_rdig[8];
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    const uint32_t warp = warp_uniform(threadIdx.x / 32u), lane = threadIdx.x % 32u;
    unsigned char* const stages = S.take(32u * kDecStage);
    unsigned char* const ctls = S.take(32u * kDecCtl);
    if (!S.ok) { if (threadIdx.x == 0) atomicOr(&ws.ctrl->err, 4u); return; }
    const uint32_t stage_s = (uint32_t)__cvta_generic_to_shared(stages) + warp * kDecStage;
    const uint32_t bar_s = (uint32_t)__cvta_generic_to_shared(ctls) + warp * kDecCtl, buf_s = bar_s + kDecBuf;
    // (a warp's control block as a pointer, and the image's parts, are worked out where they are needed)
    auto buf_of = [&]() {
        uint32_t a = buf_s;
        asm volatile("" : "+r"(a));
        return static_cast<unsigned char*>(__cvta_shared_to_generic((size_t)a));
    };
    auto payload_of = [&]() {
        const unsigned char* p = wire;
        asm volatile("" : "+l"(p));
        return p + g.meta_end;
    };
    auto tab16_of = [&]() { return reinterpret_cast<const uint16_t*>(wire + 64 + 16ull * g.n_chunks); };
    const bool copies = !(g.inject & kInjectNoCopy);

    // The ragged last tile (raw; entry 0 when its chunk is absent): by the last block's last eight warps.
    if (g.tail_len && blockIdx.x == gridDim.x - 1u && warp >= 24u && tab16_of()[g.n_full_tiles] == 0xFFFFu) {
        const uint32_t t = g.n_full_tiles, tt = threadIdx.x - 768u;
        const unsigned char* src = payload_of() + *reinterpret_cast<const unsigned long long*>(wire + 64 + 16ull * chunk_of(g, t)) + ws.rel[t];
        if (MODE != 1) copy_ragged_tile(LEAVES ? reinterpret_cast<unsigned char*>(ws.tptr[t]) : dst + (uint64_t)t * kTile, src, g.tail_len, tt);
        if (MODE != 2) {
            const uint32_t v = ragged_tile_digest(S, g, stages + 24u * kDecStage, src, s_rdig, 3, tt);
            if (tt == 0) ws.dig[t] = v;
        }
    }

    auto is_ent_entry = [](uint32_t e) { return ENT != 0 && e > 0x8000u; };
    auto is_pack_entry = [](uint32_t e) { return ENT != 1 && e >= 258u && e < 512u; };
    auto blame = [&](uint32_t t, bool structure) {       // lane 0: the tile does not keep the format (step 4)
        atomicMin(&ws.ctrl->bad4_key, (unsigned long long)t * 2ull + (structure ? 1ull : 0ull));
        atomicOr(&ws.cflag[chunk_of(g, t)], CF_BAD4);
    };
    // A coded tile's first 64 bytes, word l in lane l: whether they keep the format.  Everything that follows
    // (places, lengths of copies) is made from them, so a tile whose header does not is left out.
    auto header_ok = [&](uint32_t t, uint32_t e, uint32_t hdr) -> bool {
        int verdict = 0;
        if (is_pack_entry(e)) {
            const uint32_t x = __shfl_sync(0xFFFFFFFFu, hdr, lane >> 1), d = (lane & 1u) ? x >> 16 : x & 0xFFFFu;
            const uint32_t wr = (d >> 8) & 15u, base = d & 0xFFu, chk = d >> 12;
            const bool bad = wr > 8u || chk != (((base & 15u) ^ (base >> 4) ^ wr ^ 5u) & 15u);
            const bool anybad = __any_sync(0xFFFFFFFFu, bad);
            const uint32_t sum = __reduce_add_sync(0xFFFFFFFFu, wr);
            verdict = anybad ? 1 : (258u + sum != e ? 2 : 0);
        } else if (is_ent_entry(e)) {
            const uint32_t x = __shfl_sync(0xFFFFFFFFu, hdr, 2u + ((lane >> 1) & 3u)), cnt = (lane & 1u) ? x >> 16 : x & 0xFFFFu;
            const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, lane < 8u ? cnt : 0u);
            const bool cnt_bad = __any_sync(0xFFFFFFFFu, lane < 8u && (cnt < 64u || cnt > 319u));
            const bool spare = __any_sync(0xFFFFFFFFu, lane >= 6u && lane < 16u && hdr != 0u);       // (40 bytes that carry nothing)
            verdict = (cnt_bad || ent_tile_bytes(total) != 32u * (e & 0x7FFFu)) ? 2 : spare ? 1 : 0;
        }
        if (verdict && lane == 0) blame(t, verdict == 2);
        return verdict == 0;
    };
    auto is_coded = [&](uint32_t e) { return is_pack_entry(e) || is_ent_entry(e); };

    uint32_t phase = 0;
    // The copy of share `sh` of a tile.  `at` runs through the tile: groups' planes (32-byte units) or words of
    // the streams before the share.  Returns what the share's reader needs: PACK its four descriptors, ENT
    // the words of its stream | those before it << 16, and the anchor.
    auto start_share = [&](uint32_t e, unsigned long long src, uint32_t hdr, uint32_t sh, uint32_t& at) -> uint2 {
        uint2 r = make_uint2(0u, 0u);
        const unsigned char* const p = payload_of() + src;
        const bool go = lane == 0 && phase < kStuck && copies;
        if (is_pack_entry(e)) {
            r.x = __shfl_sync(0xFFFFFFFFu, hdr, 2u * sh);
            r.y = __shfl_sync(0xFFFFFFFFu, hdr, 2u * sh + 1u);
            const uint32_t units = __dp4a(r.x & 0x0F000F00u, 0x01000100u, __dp4a(r.y & 0x0F000F00u, 0x01000100u, 0u));
            if (go) {
                mbar_expect(bar_s, 1024u + 32u * units);
                bulk_copy_at(stage_s, p + 64u + 1024u * sh, 1024u, bar_s);
                if (units) bulk_copy_at(stage_s + kDecPlanes, p + 8256u + 32u * at, 32u * units, bar_s);
            }
            at += units;
        } else if (is_ent_entry(e)) {
            const uint32_t x = __shfl_sync(0xFFFFFFFFu, hdr, 2u + (sh >> 1)), mine = (sh & 1u) ? x >> 16 : x & 0xFFFFu;
            r.x = mine | (at << 16);
            r.y = (__shfl_sync(0xFFFFFFFFu, hdr, sh >> 2) >> (8u * (sh & 3u))) & 0xFFu;
            if (go) {
                // (two words beyond the stream, which a reader may look at; the last share's: to the tile's end)
                const uint32_t len = 32u * (e & 0x7FFFu), begin = (8512u + 4u * at) & ~15u;
                const uint32_t end = sh == 7u ? len : min(len, (8512u + 4u * (at + mine + 2u) + 15u) & ~15u);
                mbar_expect(bar_s, 1024u + 32u + end - begin);
                bulk_copy_at(stage_s, p + 64u + 1024u * sh, 1024u, bar_s);
                bulk_copy_at(stage_s + kDecPlanes, p + 8256u + 32u * sh, 32u, bar_s);
                bulk_copy_at(stage_s + kDecStream, p + begin, end - begin, bar_s);
            }
            at += mine;
        } else if (e == 512u) {
            if (go) {
                mbar_expect(bar_s, kShare);
                bulk_copy_at(stage_s, p + kShare * sh, kShare, bar_s);
            }
        }
        return r;
    };

    // The tile behind ticket k (one lane).  A masked image's tickets run over its present chunks; one that falls
    // behind the end of the cache's short last chunk has no tile, and the next one is drawn.
    const uint32_t n_first = 32u * gridDim.x;            // a warp's first ticket is its place in the grid
    auto draw = [&]() { return n_first + atomicAdd(&ws.ctrl->ticket, 1u); };
    auto place_of = [&](uint32_t k, uint32_t chunk) { return chunk * g.tiles_per_chunk + (k - chunk_of(g, k) * g.tiles_per_chunk); };
    auto tile_of = [&](uint32_t k) -> uint32_t {
        if (!masked) return k < g.n_full_tiles ? k : kNone;
        while (k < n_tickets) {
            const uint32_t t = place_of(k, ws.plist[chunk_of(g, k)]);
            if (t < g.n_full_tiles) return t;
            k = draw();
        }
        return kNone;
    };
    // A tile's entry (| kFirst: the first of its chunk), where its payload begins and where it goes, asked for
    // and taken a few shares later (by lane 0's copies into the warp's 64 bytes), and then its header.
    constexpr uint32_t kFirst = 1u << 16, kUnsound = 1u << 17;
    auto ask = [&](uint32_t t) {
        if (lane != 0) return;
        unsigned char* const buf = buf_of();
        cp_async16(buf, tab16_of() + (t & ~7u));
        cp_async16(buf + 16, ws.rel + (t & ~3u));
        cp_async16(buf + 32, wire + 64 + 16ull * chunk_of(g, t));
        if (LEAVES) cp_async16(buf + 48, ws.tptr + (t & ~1u));
    };
    auto take = [&](uint32_t t) -> uint32_t {
        cp_async_wait_all();
        __syncwarp();
        const uint32_t e = warp_uniform(lds_now_u16(buf_s + 2u * (t & 7u)));
        const uint2 po = lds_now_v2<32>(buf_s);
        const unsigned long long src = (po.x | ((unsigned long long)po.y << 32)) + lds_now<16>(buf_s + 4u * (t & 3u));
        uint2 d = make_uint2(0u, 0u);
        if (LEAVES) d = lds_now_v2<48>(buf_s + 8u * (t & 1u));
        __syncwarp();
        if (lane == 0) {
            sts_now(bar_s + kDecSrc, (uint32_t)src); sts_now(bar_s + kDecSrc + 4u, (uint32_t)(src >> 32));
            if (LEAVES) { sts_now(bar_s + kDecDst, d.x); sts_now(bar_s + kDecDst + 4u, d.y); }
        }
        if (is_coded(e) && lane < 4u) cp_async16(buf_of() + 16u * lane, payload_of() + src + 16u * lane);
        return e | (first_in_chunk(g, t) ? kFirst : 0u);
    };
    auto header_word = [&]() { return lane < 16u ? lds_now<0>(buf_s + 4u * lane) : 0u; };
    auto take_header = [&](uint32_t t, uint32_t ew) -> uint32_t {
        if (!is_coded(ew & 0xFFFFu)) return ew;
        cp_async_wait_all();
        __syncwarp();
        return header_ok(t, ew & 0xFFFFu, header_word()) ? ew : ew | kUnsound;
    };
    auto prepared = [&](uint32_t at) -> unsigned long long {
        const uint2 v = lds_now_v2<0>(bar_s + at);
        return v.x | ((unsigned long long)v.y << 32);
    };

    if (lane == 0) mbar_init(reinterpret_cast<unsigned long long*>(buf_of() - kDecBuf), 1);
    uint32_t t = kNone, ew = 0, hdr = 0, at = 0;
    unsigned long long src = 0, o_leaf = 0;
    uint2 dd = make_uint2(0u, 0u);
    if (lane == 0) t = tile_of(warp * gridDim.x + blockIdx.x);
    t = warp_uniform(__shfl_sync(0xFFFFFFFFu, t, 0));
    // the prepared tile's first copy
    auto start_tile = [&](uint32_t ew) {
        hdr = header_word();
        src = prepared(kDecSrc);
        at = 0;
        if (!(ew & kUnsound)) dd = start_share(ew & 0xFFFFu, src, hdr, 0u, at);
    };
    if (t != kNone) {
        ask(t);
        ew = take(t);
        ew = take_header(t, ew);
        __syncwarp();
        start_tile(ew);
    }
    while (t != kNone) {
        const uint32_t e = ew & 0xFFFFu;
        bool good = (ew & kUnsound) == 0u;
        const bool is_ent = is_ent_entry(e), is_coded_now = is_coded(e), started = is_coded_now ? good : e == 512u;
        if (LEAVES) o_leaf = prepared(kDecDst);
        uint32_t st = 0, tn = kNone, ewn = 0;
#pragma unroll 1
        for (uint32_t s = 0; s < 8u; s++) {
            // ---- the share's bytes into registers
            uint32_t w[kWordsPerLane];
            uint2 sm[4];
            PlaneWords pw[4];
            const uint2 dc = dd;
            bool share_ok = good;
            const uint32_t sm_s = stage_s + 8u * lane;
            const bool all4 = !is_ent && is_coded_now && all_of_width_4(dc);
            if (started) {
                wait_for_copy_at<true>(bar_s, phase, g.wait_ns, ws.ctrl, !copies);
                phase ^= 1u;
                if (!is_coded_now) {
                    read_staged_words_at(stage_s, 0u, lane, w);
                } else {
                    sm[0] = lds_now_v2<0>(sm_s); sm[1] = lds_now_v2<256>(sm_s); sm[2] = lds_now_v2<512>(sm_s); sm[3] = lds_now_v2<768>(sm_s);
                    if (is_ent) {
                        const uint32_t mine = dc.x & 0xFFFFu, before = dc.x >> 16, stream = stage_s + kDecStream + 4u * (before & 3u);
                        uint32_t eb[8];
                        bool ok = read_strands(stream, 64u + lds_now_u8(stage_s + kDecPlanes + lane), mine, dc.y, lane, ptab_s, eb);
                        if (s == 7u) {               // the fill behind the last stream
                            const uint32_t n_fill = (32u * (e & 0x7FFFu) - 8512u) / 4u - before - mine;
                            const uint32_t x = lane < n_fill ? lds_now<0>(stream + 4u * (mine + lane)) : 0u;
                            ok = !__any_sync(0xFFFFFFFFu, x != 0u) && ok;
                        }
                        if (!ok) {
                            if (lane == 0) blame(t, false);
                            share_ok = good = false;
                        }
#pragma unroll
                        for (int j = 0; j < 4; j++) { pw[j].a = eb[2 * j]; pw[j].b = eb[2 * j + 1]; }
                    } else if (ENT != 1) {
                        uint32_t rec = stage_s + kDecPlanes;
                        if (all4) {                  // (what most shares are: the planes' places are fixed)
                            rec += 4u * lane;
                            pw[0].a = lds_now<0>(rec); pw[1].a = lds_now<128>(rec); pw[2].a = lds_now<256>(rec); pw[3].a = lds_now<384>(rec);
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; j++) {
                                const uint32_t wd = ((j < 2 ? dc.x : dc.y) >> ((j & 1) ? 24 : 8)) & 15u;
                                pw[j] = read_group_planes(rec, wd, 4u * lane, 2u * lane, lane);
                                rec += 32u * wd;
                            }
                        }
                    }
                }
            } else if (e == 1u || e == 2u) {
                // a tile of zeros (nothing was shipped) or of one value (the first two bytes of its 32; the other
                // 30 are zero)
                uint32_t v = 0;
                if (e == 2u) {
                    const uint32_t x = lane < 8u ? __ldg(reinterpret_cast<const uint32_t*>(payload_of() + src) + lane) : 0u;
                    v = (__shfl_sync(0xFFFFFFFFu, x, 0) & 0xFFFFu) * 0x10001u;
                    if (__any_sync(0xFFFFFFFFu, (lane == 0u ? x >> 16 : x) != 0u)) {
                        share_ok = good = false;
                        if (lane == 0) blame(t, false);
                    }
                }
#pragma unroll
                for (int i = 0; i < 16; i++) w[i] = v;
            }
            __syncwarp();                            // the stage is free

            // ---- the next share's copy, and a step of what the next tile needs
            if (s < 7u) {
                if (started) dd = start_share(e, src, hdr, s + 1u, at);
                if (s == 0u) {
                    if (lane == 0) tn = draw();
                } else if (s == 1u) {
                    if (lane == 0 && masked && tn < n_tickets) cp_async4(buf_of(), ws.plist + chunk_of(g, tn));
                } else if (s == 2u) {
                    if (lane == 0) {
                        if (masked && tn < n_tickets) {
                            cp_async_wait_all();
                            tn = place_of(tn, lds_now<0>(buf_s));
                            if (tn >= g.n_full_tiles) tn = tile_of(draw());
                        } else if (masked || tn >= g.n_full_tiles) {
                            tn = kNone;
                        }
                    }
                    tn = warp_uniform(__shfl_sync(0xFFFFFFFFu, tn, 0));
                    if (tn != kNone) ask(tn);
                } else if (s == 4u) {
                    if (tn != kNone) ewn = take(tn);
                } else if (s == 6u) {
                    if (tn != kNone) ewn = take_header(tn, ewn);
                }
            } else if (tn != kNone) {
                start_tile(ewn);
            }

            // ---- words, stores, checksum
            if (e != 0u && share_ok) {
                unsigned char* const q = (LEAVES ? reinterpret_cast<unsigned char*>(o_leaf) : dst + (uint64_t)t * kTile) + (kShare * s + 4u * lane);
                const uint32_t how = !LEAVES ? 0u : ((uint32_t)o_leaf & 3u) == 0u ? 0u : ((uint32_t)o_leaf & 1u) ? 2u : 1u;
                // (once per way of storing: in leaf mode a tile may start off a four-byte boundary)
                auto rest_of_step = [&](auto how_c) {
                constexpr uint32_t HOW = decltype(how_c)::value;
                auto put = [&](int i, uint32_t v) {
                    if (HOW == 0u) st_stream_u32(q + i * 128, v);
                    else if (HOW == 1u) { stg_u16(q + i * 128, v); stg_u16(q + i * 128 + 2, v >> 16); }
                    else { stg_u8(q + i * 128, v); stg_u16(q + i * 128 + 1, v >> 8); stg_u8(q + i * 128 + 3, v >> 24); }
                };
                // (a tile's first state is 0, which stays 0; the all-ones start value complements a chunk's first word)
                if (MODE != 2) st = chain_step(S, st) ^ ((s == 0u && lane == 0u && (ew & kFirst)) ? 0xFFFFFFFFu : 0u);
                if (is_coded_now) {
                    auto groups = [&](auto all4_c) {
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        uint32_t ea, eb, w4[4];
                        if (ENT == 1 || (ENT == 2 && is_ent)) {
                            ea = pw[j].a; eb = pw[j].b;
                        } else {
                            const uint32_t dw = j < 2 ? dc.x : dc.y;
                            const uint32_t base = (j & 1) ? (dw >> 16) & 0xFFu : dw & 0xFFu, wd = ((j & 1) ? dw >> 24 : dw >> 8) & 15u;
                            if (decltype(all4_c)::value) {
                                unpack_nibbles(pw[j].a, ea, eb);
                                ea += base * 0x01010101u; eb += base * 0x01010101u;
                            } else {
                                unpack_group(pw[j], base, wd, ea, eb);
                            }
                        }
                        join_group(sm[j], ea, eb, w4);
                        if (MODE != 1) { put(4 * j, w4[0]); put(4 * j + 1, w4[1]); put(4 * j + 2, w4[2]); put(4 * j + 3, w4[3]); }
                        if (MODE != 2) {
                            st = chain_step(S, st ^ w4[0]);
                            st = chain_step(S, st ^ w4[1]);
                            st = chain_step(S, st ^ w4[2]);
                            st = j < 3 ? chain_step(S, st ^ w4[3]) : st ^ w4[3];
                        }
                    }
                    };
                    if (ENT != 1 && HOW != 2u && all4) groups(std::true_type());      // (byte stores: rare)
                    else groups(std::false_type());
                } else {
                    // (digest first, then the stores: see the team's loop)
                    if (MODE != 2) {
#pragma unroll
                        for (int i = 0; i < 16; i++) st = i < 15 ? chain_step(S, st ^ w[i]) : st ^ w[i];
                    }
                    if (MODE != 1) {
#pragma unroll
                        for (int i = 0; i < 16; i++) put(i, w[i]);
                    }
                }
                };
                if (!LEAVES || how == 0u) rest_of_step(std::integral_constant<uint32_t, 0u>());
                else if (how == 1u) rest_of_step(std::integral_constant<uint32_t, 1u>());
                else rest_of_step(std::integral_constant<uint32_t, 2u>());
            }
        }
        if (MODE != 2 && e != 0u && good) {
            const uint32_t v = __reduce_xor_sync(0xFFFFFFFFu, lane_finish(S, st));
            if (lane == 0) ws.dig[t] = v;
        }
        t = tn; ew = ewn;
    }
}

}  // namespace wm
