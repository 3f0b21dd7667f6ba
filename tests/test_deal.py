"""How a decode call of a masked image shares out its tiles (csrc/wm_deal.h), compiled for the host: wherever the
list of present chunks has the cache's short last chunk, every tile is some team's, once, and no team's
loop ends before one of its tiles."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "wm_deal.h"
// teams in the given order: a team runs `stride` steps before the next one's turn (0: to its end before the next one starts)
static bool run(bool in_line, uint32_t teams, uint32_t tpc, const std::vector<uint32_t>& list, uint32_t n_full, uint32_t stride, bool backwards)
{
    const uint32_t n_tickets = (uint32_t)list.size() * tpc, none = 0xFFFFFFFFu;
    uint32_t ticket = 0;
    std::vector<int> seen(n_full, 0);
    auto tile_of = [&](uint32_t k) { return list.at(k / tpc) * tpc + k % tpc; };
    auto draw = [&]() { return 3u * teams + ticket++; };
    struct Team { std::vector<uint32_t> slot; uint32_t it = 0; bool done = false; };
    std::vector<Team> team(teams);
    auto start = [&](uint32_t k) {
        const wm::FirstTiles f = in_line ? wm::deal_first_tiles_inline(k, teams, n_tickets, n_full, true, tile_of, draw)
                                         : wm::deal_first_tiles(k, teams, n_tickets, n_full, tile_of, draw);
        team[k].slot = {f.a, f.b, f.c};
    };
    auto step = [&](uint32_t k) {        // as the kernel's loop: the ticket three ahead while the tile two ahead is one
        Team& m = team[k];
        const uint32_t t = m.slot[m.it];
        if (t >= n_full) {
            for (uint32_t i = m.it; i < m.slot.size(); i++) if (m.slot[i] < n_full) return false;
            return m.done = true;
        }
        seen[t]++;
        uint32_t next = none;
        if (m.slot[m.it + 2] < n_full)
            for (uint32_t d = draw(); d < n_tickets; d = draw())
                if (tile_of(d) < n_full) { next = tile_of(d); break; }
        m.slot.push_back(next);
        m.it++;
        return true;
    };
    auto at = [&](uint32_t i) { return backwards ? teams - 1 - i : i; };
    if (stride == 0) {
        for (uint32_t i = 0; i < teams; i++) { start(at(i)); while (!team[at(i)].done) if (!step(at(i))) return false; }
    } else {
        for (uint32_t i = 0; i < teams; i++) start(at(i));
        for (bool any = true; any;) {
            any = false;
            for (uint32_t i = 0; i < teams; i++)
                for (uint32_t s = 0; s < stride && !team[at(i)].done; s++) { any = true; if (!step(at(i))) return false; }
        }
    }
    for (uint32_t c : list)
        for (uint32_t t = c * tpc; t < (c + 1) * tpc; t++)
            if (t < n_full && seen[t]-- != 1) return false;
    for (int v : seen) if (v) return false;
    return true;
}
int main(int, char** argv)
{
    const uint32_t tpc = atoi(argv[1]), rest = atoi(argv[2]);         // full tiles of the last chunk
    const bool in_line = atoi(argv[3]) != 0;
    uint32_t runs = 0;
    for (uint32_t chunks = 1; chunks <= 7; chunks++)
        for (uint32_t skip = 1; skip <= 2; skip++)                    // every chunk, every other one
            for (uint32_t place = 0; place < chunks; place++) {       // where the list has the last chunk
                std::vector<uint32_t> list;
                for (uint32_t i = 0; i + 1 < chunks; i++) list.push_back(i * skip);
                const uint32_t last = (chunks - 1) * skip;
                list.insert(list.begin() + place, last);
                for (uint32_t teams = 1; teams <= chunks * tpc + 1; teams++)
                    for (uint32_t stride : {0u, 1u, 3u})
                        for (bool backwards : {false, true}) {
                            runs++;
                            if (!run(in_line, teams, tpc, list, last * tpc + rest, stride, backwards)) {
                                printf("chunks %u skip %u place %u teams %u stride %u %d\n", chunks, skip, place, teams, stride, (int)backwards);
                                return 1;
                            }
                        }
            }
    printf("%u runs\n", runs);
    return runs ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("deal")
    (d / "deal.cpp").write_text(PROGRAM)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-I", os.path.join(ROOT, "paper_2607_10389_b200", "csrc"),
                           str(d / "deal.cpp"), "-o", str(d / "deal")])
    return str(d / "deal")


@pytest.mark.parametrize("tiles_per_chunk,rest", [(1, 0), (1, 1), (3, 0), (3, 1), (3, 2), (4, 0), (4, 1), (4, 4), (16, 0), (16, 1), (16, 13)])
@pytest.mark.parametrize("in_line", [0, 1])
def test_every_tile_is_decoded_once(program, tiles_per_chunk, rest, in_line):
    out = subprocess.run([program, str(tiles_per_chunk), str(rest), str(in_line)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
