"""Grid independence: tiles are claimed by ticket, so the wire image, the CRC vector and every
result are the same whatever number of thread blocks the main kernels run on.  WM_OPT_BLOCKS caps
that number for callers that share the GPU; here it also serves to prove the independence
(1 encoding block beside the scanner, a handful, half the machine, all of it, more than exist)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_10389_b200 import binding as wm
from paper_2607_10389_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("options,kw", [(0, {}), (wm.OPT_ENTROPY, {"entropy": True}),
                                        (wm.OPT_ZERO_TILES | wm.OPT_ENTROPY, {"entropy": True, "zero_tiles": True})])
def test_same_bytes_at_every_block_count(options, kw):
    cfg = inputs.CONFIGS["engine_small"]
    host = inputs.make_cache(cfg)[: cfg.nbytes - 1234].contiguous()
    host[5 * 65536: 5 * 65536 + 3 * 16384] = 0
    chunk = 65536
    cur = host.cuda()
    n = cur.numel()
    nc = wm.num_chunks(n, chunk)
    rng = np.random.default_rng(11)
    for mask in (None, (rng.random(nc) < 0.75).astype(np.uint8)):
        crc_in = rng.integers(0, 2**32, nc, dtype=np.uint64).astype(np.uint32)
        want_wire, want_crc, want = oracle.encode(host.numpy(), chunk, dirty=mask, crc_in=crc_in, **kw)
        d = None if mask is None else torch.from_numpy(mask).cuda()
        ws, res = wm.new_workspace(n, chunk), wm.new_result()
        wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
        for blocks in (0, 2, 3, 37, 74, 148, 255):
            crc = torch.from_numpy(crc_in.view(np.int32).copy()).cuda()
            wire.fill_(0xEE)
            wm.wm_encode_opt(cur, chunk, d, crc, wire, ws, res, options | wm.opt_blocks(blocks))
            r = wm.read_result(res)
            assert r.ok and (r.wire_len, r.cache_crc, r.n_present) == (want.wire_len, want.cache_crc, want.n_present), blocks
            assert np.array_equal(wire[: r.wire_len].cpu().numpy(), want_wire), blocks
            assert np.array_equal(crc.cpu().numpy().view(np.uint32), want_crc), blocks
        for blocks in (0, 1, 2, 37, 74, 255):
            dst = host.cuda() if mask is not None else torch.zeros(n, dtype=torch.uint8, device="cuda")
            dst_crc = torch.from_numpy(want_crc.view(np.int32).copy()).cuda() if mask is not None else \
                torch.zeros(nc, dtype=torch.int32, device="cuda")
            wm.wm_decode_verify_opt(wire, r.wire_len, dst, chunk, dst_crc, ws, res,
                                    (options & wm.OPT_ENTROPY) | wm.opt_blocks(blocks))
            rd = wm.read_result(res)
            assert rd.ok and torch.equal(dst, cur), blocks
            assert np.array_equal(dst_crc.cpu().numpy().view(np.uint32), want_crc), blocks


def test_a_block_cap_of_one_is_refused_for_encode():
    cur = torch.zeros(65536, dtype=torch.uint8, device="cuda")
    ws, res = wm.new_workspace(65536, 65536), wm.new_result()
    wire = torch.zeros(wm.wire_bound(65536, 65536), dtype=torch.uint8, device="cuda")
    crc = torch.zeros(1, dtype=torch.int32, device="cuda")
    with pytest.raises(wm.WmError, match="ERR_ARG"):
        wm.wm_encode_opt(cur, 65536, None, crc, wire, ws, res, wm.opt_blocks(1))


def test_placement_is_repeatable_over_many_moves_and_block_counts():
    """Which team gets which tile first changes from run to run and with the number of blocks; the
    bytes must not.  400 moves of a 64 MiB cache, every option set, block counts drawn at random:
    every image equals the first of its option set byte for byte, every round trip returns the
    cache, and no call ends in a timeout."""
    cfg = inputs.CONFIGS["engine_small"]
    g = torch.Generator(device="cuda").manual_seed(77)
    n, chunk = 64 << 20, 1 << 20
    cur = (torch.randn(n // 2, generator=g, device="cuda") * 3).to(torch.bfloat16).view(torch.uint8)
    cur[5 << 20: 6 << 20] = 0
    nc = wm.num_chunks(n, chunk)
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    dst = torch.zeros(n, dtype=torch.uint8, device="cuda")
    dcrc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    rng = np.random.default_rng(5)
    first = {}
    for i in range(400):
        opt = int(rng.integers(0, 4))
        be, bd = int(rng.choice([0, 2, 5, 37, 74, 111, 148])), int(rng.choice([0, 1, 5, 37, 74, 111, 148]))
        wm.wm_encode_opt(cur, chunk, None, crc, wire, ws, res, opt | wm.opt_blocks(be))
        r = wm.read_result(res)
        assert r.ok, (i, r.status_name)
        img = wire[: r.wire_len]
        if opt not in first:
            first[opt] = (img.clone(), crc.clone())
        assert torch.equal(img, first[opt][0]) and torch.equal(crc, first[opt][1]), (i, opt, be)
        if i % 4 == 0:
            wm.wm_decode_verify_opt(wire, r.wire_len, dst, chunk, dcrc, ws, res, (opt & wm.OPT_ENTROPY) | wm.opt_blocks(bd))
            assert wm.read_result(res).ok and torch.equal(dst, cur) and torch.equal(dcrc, crc), (i, opt, bd)


@pytest.mark.parametrize("chunk_tiles", [1, 3, 4])
@pytest.mark.parametrize("options,kw", [(0, {}), (wm.OPT_ENTROPY | wm.OPT_ZERO_TILES, {"entropy": True, "zero_tiles": True})])
def test_sparse_and_degenerate_masks(chunk_tiles, options, kw):
    """Masked calls claim only the tiles of present chunks.  The masks that stress that: nothing
    present, everything present (with the mask flag), only the short last chunk, everything but
    the last chunk, single chunks, every other chunk; chunk sizes of 1, 3 (no power of two) and
    4 tiles on a cache whose last chunk and last tile are ragged.  Image, CRC vector and result
    are the oracle's; the decode installs exactly the present chunks."""
    TILE = 16384
    chunk = chunk_tiles * TILE
    cfg = inputs.CONFIGS["engine_small"]
    host = inputs.make_cache(cfg)[: 41 * TILE + 777].contiguous()
    host[7 * TILE: 9 * TILE] = 0
    cur = host.cuda()
    n = cur.numel()
    nc = wm.num_chunks(n, chunk)
    masks = {"none": np.zeros(nc, np.uint8), "all": np.ones(nc, np.uint8)}
    m = np.zeros(nc, np.uint8); m[-1] = 1; masks["last only"] = m
    m = np.ones(nc, np.uint8); m[-1] = 0; masks["all but last"] = m
    m = np.zeros(nc, np.uint8); m[0] = 1; masks["first only"] = m
    m = np.zeros(nc, np.uint8); m[nc // 2] = 1; masks["one in the middle"] = m
    masks["every other"] = (np.arange(nc) % 2).astype(np.uint8)
    masks["every other, and the last"] = ((np.arange(nc) % 2 == 0) | (np.arange(nc) == nc - 1)).astype(np.uint8)
    rng = np.random.default_rng(1)
    crc_in = rng.integers(0, 2**32, nc, dtype=np.uint64).astype(np.uint32)
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
    old = torch.full((n,), 0x3C, dtype=torch.uint8, device="cuda")
    for name, mask in masks.items():
        want_wire, want_crc, want = oracle.encode(host.numpy(), chunk, dirty=mask, crc_in=crc_in, **kw)
        crc = torch.from_numpy(crc_in.view(np.int32).copy()).cuda()
        wire.fill_(0xEE)
        wm.wm_encode_opt(cur, chunk, torch.from_numpy(mask).cuda(), crc, wire, ws, res, options)
        r = wm.read_result(res)
        assert r.ok and (r.wire_len, r.cache_crc, r.n_present, r.payload_bytes) == \
            (want.wire_len, want.cache_crc, want.n_present, want.payload_bytes), name
        assert np.array_equal(wire[: r.wire_len].cpu().numpy(), want_wire), name
        assert np.array_equal(crc.cpu().numpy().view(np.uint32), want_crc), name
        dst = old.clone()
        dcrc = torch.from_numpy(want_crc.view(np.int32).copy()).cuda()
        wm.wm_decode_verify_opt(wire, r.wire_len, dst, chunk, dcrc, ws, res, options & wm.OPT_ENTROPY)
        assert wm.read_result(res).ok, name
        got = dst.cpu().numpy()
        for c in range(nc):
            lo, hi = c * chunk, min((c + 1) * chunk, n)
            if mask[c]:
                assert np.array_equal(got[lo:hi], host.numpy()[lo:hi]), (name, c)
            else:
                assert (got[lo:hi] == 0x3C).all(), (name, c)


@pytest.mark.parametrize("tiles", [1, 2, 7, 8, 147, 148, 8 * 147, 8 * 147 + 1, 2 * 8 * 148, 2 * 8 * 148 + 1])
@pytest.mark.parametrize("masked", [False, True])
def test_encode_around_the_numbers_of_teams(tiles, masked):
    """A block runs fewer of its eight teams when there are fewer tiles than teams; every team takes one tile first
    up to two tiles per team, two from there on."""
    n, chunk = tiles * 16384, 2 * 16384
    g = torch.Generator("cuda").manual_seed(tiles)
    cur = torch.randn(n // 2, generator=g, device="cuda").to(torch.bfloat16).view(torch.uint8)
    nc = wm.num_chunks(n, chunk)
    mask = np.array([c % 4 != 2 for c in range(nc)], np.uint8) if masked else None
    want_wire, want_crc, want = oracle.encode(cur.cpu().numpy(), chunk, dirty=mask, crc_in=np.zeros(nc, np.uint32))
    ws, res, crc = wm.new_workspace(n, chunk), wm.new_result(), torch.zeros(nc, dtype=torch.int32, device="cuda")
    wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
    wm.wm_encode(cur, chunk, None if mask is None else torch.from_numpy(mask).cuda(), crc, wire, ws, res)
    r = wm.read_result(res)
    assert r.ok and r.wire_len == want.wire_len and np.array_equal(wire[: r.wire_len].cpu().numpy(), want_wire)
    assert np.array_equal(crc.cpu().numpy().view(np.uint32), want_crc)


@pytest.mark.parametrize("tiles", [8 * 147 - 1, 8 * 147 + 147, 8 * 147 + 148, 12 * 147 + 5, 16 * 147, 16 * 147 + 1])
@pytest.mark.parametrize("options", [0, wm.OPT_ENTROPY])
@pytest.mark.parametrize("masked", [False, True])
def test_encode_between_one_and_two_tiles_per_team(tiles, options, masked):
    """Every block has the same number of tiles there, some teams a second one; capped at 37 blocks the same cache
    has more than that.  With a mask the cache is larger and as many of its tiles are present."""
    chunk_tiles = 1 if masked else 3
    n, chunk = (tiles * 3 // 2 if masked else tiles) * 16384 - 5, chunk_tiles * 16384
    g = torch.Generator("cuda").manual_seed(tiles + options)
    cur = torch.randn((n + 1) // 2, generator=g, device="cuda").to(torch.bfloat16).view(torch.uint8)[:n].contiguous()
    nc = wm.num_chunks(n, chunk)
    mask = np.array([c % 3 != 2 for c in range(nc)], np.uint8) if masked else None
    want_wire, want_crc, want = oracle.encode(cur.cpu().numpy(), chunk, dirty=mask, crc_in=np.zeros(nc, np.uint32), entropy=bool(options))
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    for blocks in (0, 37, 0):
        crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
        wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
        wm.wm_encode_opt(cur, chunk, None if mask is None else torch.from_numpy(mask).cuda(), crc, wire, ws, res, options | wm.opt_blocks(blocks))
        r = wm.read_result(res)
        assert r.ok and r.wire_len == want.wire_len and np.array_equal(wire[: r.wire_len].cpu().numpy(), want_wire), blocks
        assert np.array_equal(crc.cpu().numpy().view(np.uint32), want_crc), blocks


@pytest.mark.parametrize("tiles", [1, 3, 4, 5, 8, 9, 12, 13, 14, 17])
@pytest.mark.parametrize("tail", [0, 777])
@pytest.mark.parametrize("chunk_tiles", [3, 4])
def test_decode_of_one_to_four_tiles_per_team(tiles, tail, chunk_tiles):
    """One block has four teams; the first three tickets of each are dealt out.  The sizes are the edges of that;
    with a mask the last tickets may fall behind the cache's short last chunk (one warp lists these few chunks, in order)."""
    TILE = 16384
    chunk, n = chunk_tiles * TILE, tiles * TILE + tail
    host = inputs.make_cache(inputs.CONFIGS["engine_small"])[:n].contiguous()
    cur, nc = host.cuda(), wm.num_chunks(n, chunk)
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    last = np.zeros(nc, np.uint8)
    last[-1] = 1
    half = (np.arange(nc) % 2 == (nc - 1) % 2).astype(np.uint8)
    for mask in (None, np.ones(nc, np.uint8), last, half):
        crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
        wm.wm_checksum(cur, chunk, crc, ws)
        wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
        wm.wm_encode(cur, chunk, None if mask is None else torch.from_numpy(mask).cuda(), crc, wire, ws, res)
        r = wm.read_result(res)
        assert r.ok
        present = np.repeat(np.ones(nc, bool) if mask is None else mask != 0, chunk)[:n]
        start = np.where(present, 0xEE, host.numpy()).astype(np.uint8)
        for opt in (0, wm.OPT_STRICT):
            for blocks in (1, 2):
                dst, dst_crc = torch.from_numpy(start).cuda(), crc.clone()
                wm.wm_decode_verify_opt(wire, r.wire_len, dst, chunk, dst_crc, ws, res, opt | wm.opt_blocks(blocks))
                assert wm.read_result(res).ok and torch.equal(dst, cur), (opt, blocks)
                assert torch.equal(dst_crc, crc)


@pytest.mark.parametrize("rest,tail", [(1, 0), (2, 777), (0, 5)])
@pytest.mark.parametrize("leaves", [False, True])
@pytest.mark.parametrize("options", [0, wm.OPT_STRICT, wm.OPT_ENTROPY, wm.OPT_ENTROPY | wm.OPT_STRICT])
def test_masked_decode_of_few_tickets_per_team(rest, tail, leaves, options):
    """Chunks of more than 16 tiles have a warp each in the check, so the short last chunk may stand anywhere in the list of
    present chunks and its tickets without a tile among the first ones.  The block counts are around one and three tickets
    per team.  (Every place in the list, one after the other: tests/test_deal.py.)"""
    TILE, tpc = 16384, 64
    chunk, n = tpc * TILE, (3 * tpc + rest) * TILE + tail
    host = inputs.make_cache(inputs.CONFIGS["tiny8m"])[:n].contiguous()
    cur, nc = host.cuda(), wm.num_chunks(n, chunk)
    ws, res, entropy = wm.new_workspace(n, chunk), wm.new_result(), options & wm.OPT_ENTROPY
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    wm.wm_checksum(cur, chunk, crc, ws)
    cuts = [0, 3 * TILE + 100, 40 * TILE + 102, 100 * TILE + 7, n] if leaves else [0, n]
    for mask in ([1, 1, 1, 1], [0, 1, 0, 1], [0, 0, 0, 1], [1, 0, 1, 0]):
        m = np.array(mask, np.uint8)
        wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
        wm.wm_encode_opt(cur, chunk, torch.from_numpy(m).cuda(), crc.clone(), wire, ws, res, entropy)
        r = wm.read_result(res)
        assert r.ok
        start = torch.from_numpy(np.where(np.repeat(m != 0, chunk)[:n], 0xEE, host.numpy()).astype(np.uint8)).cuda()
        tickets = tpc * int(m.sum())
        for blocks in sorted({1, tickets // 12 - 1, tickets // 12, -(-tickets // 12), tickets // 4 - 1, tickets // 4} - {0}):
            for _ in range(3):
                pieces = [start[a:b].clone() for a, b in zip(cuts, cuts[1:])]
                table = wm.make_leaf_table(pieces) if leaves else None
                dst_crc = crc.clone()
                wm.wm_decode_verify_opt(wire, r.wire_len, None if leaves else pieces[0], chunk, dst_crc, ws, res, options | wm.opt_blocks(blocks),
                                        leaf_table=table, nbytes=n)
                rd = wm.read_result(res)
                assert rd.ok and torch.equal(torch.cat(pieces), cur) and torch.equal(dst_crc, crc), (mask, blocks)
