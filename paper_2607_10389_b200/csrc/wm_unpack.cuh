// From a staged tile to words: what the two loops of the decode kernel share.  Plane words and their
// unpacking (PACK tiles), a share's strands (ENT tiles), and the words put together again.
// Part of the one translation unit wm_kernels.cu (included there, in this order).
#pragma once

namespace wm {

// The plane words of one group as stored (aligned per-lane units, see pack_group):
// a = the 4-bit plane's word or the low half of an 8-bit plane; b = the 2-bit plane's 16 bits
// in the low half and the 1-bit plane's byte in bits 16-23, or the high half of an 8-bit plane.
struct PlaneWords { uint32_t a, b; };

// rec: shared-window address of the group's planes; l4 / l2 / l1: 4, 2, 1 times the lane number
__device__ __forceinline__ PlaneWords read_group_planes(uint32_t rec, uint32_t wd, uint32_t l4, uint32_t l2, uint32_t l1)
{
    PlaneWords pw;
    pw.a = 0; pw.b = 0;
    if (wd == 8u) {
        const uint2 v = lds_now_v2<0>(rec + 2u * l4);
        pw.a = v.x; pw.b = v.y;
        return pw;
    }
    if (wd & 4u) { pw.a = lds_now<0>(rec + l4); rec += 128u; }
    if (wd & 2u) { pw.b = lds_now_u16(rec + l2); rec += 64u; }
    if (wd & 1u) { pw.b |= lds_now_u8(rec + l1) << 16; }
    return pw;
}

// The eight 4-bit deltas of a plane word, one per byte (two words, coded order).
__device__ __forceinline__ void unpack_nibbles(uint32_t a, uint32_t& da, uint32_t& db)
{
    const uint32_t even = a & 0x0F0F0F0Fu, odd = (a >> 4) & 0x0F0F0F0Fu;
    da = __byte_perm(even, odd, 0x5140);
    db = __byte_perm(even, odd, 0x7362);
}

// Inverse of pack_group: the lane's eight exponent bytes (two words, coded order).  Width 4 is
// by far the most frequent; the others share one piece of code that goes plane by plane (seven
// pieces, four times each in the loop, were more than the instruction cache wants to hold).
__device__ __forceinline__ void unpack_group(const PlaneWords& pw, uint32_t base, uint32_t wd, uint32_t& ea, uint32_t& eb)
{
    uint32_t da = 0, db = 0;
    if (wd == 4u) {
        unpack_nibbles(pw.a, da, db);
    } else if (wd == 8u) {
        da = pw.a; db = pw.b;
    } else {
        if (wd & 4u) unpack_nibbles(pw.a, da, db);
        uint32_t sh = wd & 4u;
        if (wd & 2u) {      // byte -> four 2-bit fields, one per byte
            uint32_t xa = pw.b & 0xFFu, xb = (pw.b >> 8) & 0xFFu;
            xa = (xa * 0x1001u) & 0x000F000Fu; xa = (xa * 0x41u) & 0x03030303u;
            xb = (xb * 0x1001u) & 0x000F000Fu; xb = (xb * 0x41u) & 0x03030303u;
            da |= xa << sh; db |= xb << sh;
            sh += 2u;
        }
        if (wd & 1u) {      // nibble -> four bits, one per byte
            const uint32_t xa = (((pw.b >> 16) & 0xFu) * 0x00204081u) & 0x01010101u;
            const uint32_t xb = (((pw.b >> 20) & 0xFu) * 0x00204081u) & 0x01010101u;
            da |= xa << sh; db |= xb << sh;
        }
    }
    const uint32_t b4 = base * 0x01010101u;
    if (base + ((1u << wd) - 1u) <= 255u) {       // no byte can wrap: plain add
        ea = da + b4; eb = db + b4;
    } else {                                      // per byte (base + d) & 0xFF
        ea = ((da & 0x7F7F7F7Fu) + (b4 & 0x7F7F7F7Fu)) ^ ((da ^ b4) & 0x80808080u);
        eb = ((db & 0x7F7F7F7Fu) + (b4 & 0x7F7F7F7Fu)) ^ ((db ^ b4) & 0x80808080u);
    }
}

// A share whose four groups have width 4 and bases that no delta carries past 255.
__device__ __forceinline__ bool all_of_width_4(uint2 dd)
{
    const uint32_t w = ((dd.x ^ 0x04000400u) | (dd.y ^ 0x04000400u)) & 0x0F000F00u;
    const uint32_t over = (((dd.x & 0x00FF00FFu) + 0x000F000Fu) | ((dd.y & 0x00FF00FFu) + 0x000F000Fu)) & 0x01000100u;
    return (w | over) == 0u;
}

// ENT tile: lane l reads strand l of a share.  The strands lie one behind the other in the share's
// stream (`st`: the shared-window address of its first word, `mine` words long) and their lengths are
// written down (`nb`: this lane's, in bits), so a prefix sum over the lanes gives every lane the bit
// where its strand starts, and from there it reads its 32 codewords through a 64-bit window that is
// refilled a word at a time before every second codeword.  No lane waits for another.  ew: the
// exponent bytes in coded order.  False when the stream breaks a rule of the format: the lengths do not
// add up to the stream, 32 codewords do not take a strand's length, bits behind the last strand are set,
// the anchor is not the rounded mean of the share's exponents.
__device__ __forceinline__ bool read_strands(uint32_t st, uint32_t nb, uint32_t mine, uint32_t anchor, uint32_t lane, uint32_t ptab_s, uint32_t (&ew)[8])
{
    uint32_t incl = nb;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= (uint32_t)d) incl += o;
    }
    const uint32_t share_bits = __shfl_sync(0xFFFFFFFFu, incl, 31);
    if (((share_bits + 31u) >> 5) != mine) return false;
    const uint32_t start = incl - nb, wi = start >> 5, sh = start & 31u;
    // (a strand that runs past its length only fails the check below: no word beyond
    // the share's last two is ever read)
    // The window: lo holds the next 32 bits of the strand, hi what follows, `avail` of the
    // 64 are real.  (PTX shifts clamp at 32, which is what the edge cases need.)
    uint32_t lo = lds_now<0>(st + 4u * wi), hi = lds_now<4>(st + 4u * wi);
    lo = __funnelshift_r(lo, hi, sh);
    hi >>= sh;
    uint32_t avail = 64u - sh, next = wi + 2u;
#pragma unroll
    for (int j = 0; j < 8; j++) ew[j] = 0u;
#pragma unroll
    for (int i = 0; i < 32; i++) {
        if ((i & 1) == 0 && avail <= 32u) {      // (two codewords take 32 bits at most)
            const uint32_t w = lds_now<0>(st + 4u * min(next, mine + 1u));
            lo |= shl_clamp(w, avail);
            hi = shr_clamp(w, 32u - avail);
            avail += 32u;
            next++;
        }
        const uint32_t at = (lo & 0xFFu) | ptab_s;
        const uint32_t len = lds_tab_u8(at);
        const uint32_t E = len == 16u ? lo >> 8 : anchor + lds_tab_u8(at + 256u);      // (its low byte)
        ew[i >> 2] = __byte_perm(ew[i >> 2], E, (i & 3) == 0 ? 0x3214 : (i & 3) == 1 ? 0x3240 : (i & 3) == 2 ? 0x3410 : 0x4210);
        lo = __funnelshift_r(lo, hi, len);
        hi >>= len;
        avail -= len;
    }
    // the 32 codewords took exactly the strand's length; behind the last strand the
    // stream's last word is zero
    const uint32_t used = 32u * (next - wi) - sh - avail;
    const uint32_t fill = 32u * mine - share_bits;
    const bool fill_bad = lane == 31u && (lo & ((1u << fill) - 1u)) != 0u;
    // the anchor must be what the encoder writes: the rounded mean of the share's exponents
    // (otherwise the anchor of a share that holds escapes only could change unnoticed)
    uint32_t esum = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) esum = __dp4a(ew[j], 0x01010101u, esum);
    const bool anchor_ok = ((__reduce_add_sync(0xFFFFFFFFu, esum) + 512u) >> 10) == anchor;
    return !__any_sync(0xFFFFFFFFu, used != nb || fill_bad) && anchor_ok;
}

// A group's four words of this lane from its sign-mantissa bytes and its exponent bytes.  A word rotated
// left by one bit reads [E | m << 1 | sign of the other half] in each half: swap bit 0 inside the byte
// pairs of the sign-mantissa words, put the exponent bytes beside them, rotate back.
__device__ __forceinline__ void join_group(uint2 sm, uint32_t ea, uint32_t eb, uint32_t (&w)[4])
{
    const uint32_t xa = __byte_perm(sm.x, sm.x, 0x2301), xb = __byte_perm(sm.y, sm.y, 0x2301);
    const uint32_t sa = (sm.x & 0xFEFEFEFEu) | (xa & 0x01010101u), sb = (sm.y & 0xFEFEFEFEu) | (xb & 0x01010101u);
    const uint32_t r0 = __byte_perm(sa, ea, 0x5140), r1 = __byte_perm(sa, ea, 0x7362);
    const uint32_t r2 = __byte_perm(sb, eb, 0x5140), r3 = __byte_perm(sb, eb, 0x7362);
    w[0] = __funnelshift_r(r0, r0, 1); w[1] = __funnelshift_r(r1, r1, 1);
    w[2] = __funnelshift_r(r2, r2, 1); w[3] = __funnelshift_r(r3, r3, 1);
}

}  // namespace wm
