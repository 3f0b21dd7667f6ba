// The tiles of a decode team's first three steps when the image has a dirty mask.  Plain C++, for the
// kernel and for a test on the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define WM_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define WM_HOST_DEVICE inline
#endif

namespace wm {

struct FirstTiles { uint32_t a, b, c; };       // of steps 0, 1 and 2 (0xFFFFFFFF: none)

// Team k of `teams` is dealt the tickets k, k + teams and k + 2 teams.  A ticket may have no tile (tile_of
// says n_full or more): the last chunk of the cache is shorter than the others and stands anywhere in
// the list.  In its place one is drawn, until a ticket with a tile or the tickets' end.  A step without a
// tile ends the team's loop, so none stands before one that has a tile.
template <typename TileOf, typename Draw>
WM_HOST_DEVICE FirstTiles deal_first_tiles(uint32_t k, uint32_t teams, uint32_t n_tickets, uint32_t n_full, TileOf tile_of, Draw draw)
{
    constexpr uint32_t kNoTile = 0xFFFFFFFFu;
    FirstTiles f = {kNoTile, kNoTile, kNoTile};
#ifdef __CUDACC__
#pragma unroll 1
#endif
    for (uint32_t i = 0; i < 3u && k < n_tickets; i++, k += teams) {
        uint32_t t = tile_of(k);
        while (t >= n_full) {
            const uint32_t d = draw();
            if (d >= n_tickets) break;
            t = tile_of(d);
        }
        if (t >= n_full) continue;
        if (f.a == kNoTile) f.a = t; else if (f.b == kNoTile) f.b = t; else f.c = t;
    }
    return f;
}

// The same without a loop, for images with and without a mask (without one a ticket is its tile's number, and all
// tickets have tiles); a call of a ticket per team is its first case.
template <typename TileOf, typename Draw>
WM_HOST_DEVICE FirstTiles deal_first_tiles_inline(uint32_t k, uint32_t teams, uint32_t n_tickets, uint32_t n_full, bool masked, TileOf tile_of, Draw draw)
{
    constexpr uint32_t kNoTile = 0xFFFFFFFFu;
    auto dealt = [&](uint32_t kk) -> uint32_t {
        if (kk >= n_tickets) return kNoTile;
        uint32_t t = tile_of(kk);
        if (!masked || t < n_full) return t;
        for (uint32_t d = draw(); d < n_tickets; d = draw()) {
            t = tile_of(d);
            if (t < n_full) return t;
        }
        return kNoTile;
    };
    FirstTiles f = {kNoTile, kNoTile, kNoTile};
    if (n_tickets <= teams) {
        if (k < n_tickets) f.a = tile_of(k);
    } else {
        f.a = dealt(k); f.b = dealt(k + teams); f.c = dealt(k + 2u * teams);
    }
    if (masked && f.b == kNoTile) { f.b = f.c; f.c = kNoTile; }
    if (masked && f.a == kNoTile) { f.a = f.b; f.b = f.c; f.c = kNoTile; }
    return f;
}

}  // namespace wm
