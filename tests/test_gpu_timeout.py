"""The give-up paths, run for real: every device-side wait is bounded by time, and when the bound
passes the kernels return, the call reports ERR_TIMEOUT, nothing is installed, nothing is written
out of bounds, and the next call on the same workspace works.

No fault and no hang is involved: the test hook wm_inject_stall leaves out what the waits wait
for (the encode kernel's scanner, the bulk copies of the checksum and decode kernels), and a short
budget (wm_wait_budget_ms) lets the waits run out after a few tens of milliseconds.
"""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2607_10389_b200 import binding as wm
from paper_2607_10389_b200 import inputs

pytestmark = pytest.mark.gpu

BUDGET_MS = 40


@pytest.fixture
def stalled():
    """Calls issued inside the `with stalled():` block time out; outside it they run normally."""
    class Ctx:
        def __init__(self, what=True):
            self.what = what

        def __enter__(self):
            wm.wait_budget_ms(BUDGET_MS)
            wm.inject_stall(self.what)

        def __exit__(self, *a):
            torch.cuda.synchronize()
            wm.inject_stall(False)
            wm.wait_budget_ms(2000)
    yield Ctx
    wm.inject_stall(False)
    wm.wait_budget_ms(2000)


def _cache():
    cfg = inputs.CONFIGS["tiny8m"]
    host = inputs.make_cache(cfg)[: cfg.nbytes - 4321].contiguous()      # ragged tail
    return host, host.cuda(), cfg.chunk_bytes


def test_encode_gives_up_when_no_offset_ever_comes(stalled):
    host, cur, chunk = _cache()
    n = cur.numel()
    nc = wm.num_chunks(n, chunk)
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    cap = wm.wire_bound(n, chunk)
    wire = torch.full((cap + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    t0 = time.time()
    with stalled():
        wm.wm_encode(cur, chunk, None, crc, wire, ws, res, wire_cap=cap)
        r = wm.read_result(res)
    assert r.status_name == "ERR_TIMEOUT"
    assert time.time() - t0 < 20                                     # bounded: the budget, not a hang
    assert wm.workspace_status(ws) == -10
    assert bool((wire[cap:] == 0xA5).all()), "wrote past wire_cap"
    # the same workspace, wire and result record right afterwards, no clean-up in between
    wm.wm_encode(cur, chunk, None, crc, wire, ws, res, wire_cap=cap)
    r = wm.read_result(res)
    want_wire, want_crc, want = oracle.encode(host.numpy(), chunk)
    assert r.ok and r.wire_len == want.wire_len and wm.workspace_status(ws) == 0
    assert np.array_equal(wire[: r.wire_len].cpu().numpy(), want_wire)
    assert np.array_equal(crc.cpu().numpy().view(np.uint32), want_crc)


@pytest.mark.parametrize("options", [0, wm.OPT_ENTROPY])
@pytest.mark.parametrize("masked", [False, True])
def test_encode_gives_up_with_several_tiles_per_team(stalled, options, masked):
    """When one team gives up for the call, the others have copies on their way into their stages: a team has to wait
    for its own before it starts another on the same barrier, and before its block ends."""
    n, chunk = 4000 * 16384 + 7777, 8 * 16384
    cur = torch.randn((n + 1) // 2, generator=torch.Generator("cuda").manual_seed(3), device="cuda").to(torch.bfloat16).view(torch.uint8)[:n].contiguous()
    nc, cap = wm.num_chunks(n, chunk), wm.wire_bound(n, chunk)
    mask = (torch.arange(nc, device="cuda") % 8 != 3).to(torch.uint8) if masked else None
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    wire = torch.full((cap + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")

    def encode():
        wm.wm_encode_opt(cur, chunk, mask, crc, wire[:cap], ws, res, options)
        return wm.read_result(res)
    r = encode()
    want, want_crc = wire[: r.wire_len].clone(), crc.clone()
    assert r.ok
    for _ in range(3):
        t0 = time.time()
        with stalled():
            bad = encode()
        assert bad.status_name == "ERR_TIMEOUT" and time.time() - t0 < 20
        assert bool((wire[cap:] == 0xA5).all()), "wrote past wire_cap"
        crc.zero_()
        r = encode()
        assert r.ok and torch.equal(wire[: r.wire_len], want) and torch.equal(crc, want_crc)


@pytest.mark.parametrize("options", [0, wm.OPT_ENTROPY, wm.OPT_ZERO_TILES])
@pytest.mark.parametrize("tiles", [1, 3000])
def test_encode_publishes_raw_lengths_when_the_widths_never_count_as_complete(stalled, options, tiles):
    """A length that is published without its tile's widths must hold whatever they turn out to be, or the packing
    step writes more than was checked against the room in the wire buffer: the tile has to be published as raw."""
    n, chunk = tiles * 16384, 8 * 16384
    g = torch.Generator("cuda").manual_seed(tiles + options)
    cur = torch.randn(n // 2, generator=g, device="cuda").to(torch.bfloat16).view(torch.uint8)
    cur[n // 2:].random_(0, 256, generator=g)                        # half of it incompressible
    nc, meta = wm.num_chunks(n, chunk), wm.meta_bytes(n, chunk)
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    wire = torch.full((wm.wire_bound(n, chunk) + 65536,), 0xA5, dtype=torch.uint8, device="cuda")
    wm.wm_encode_opt(cur, chunk, None, crc, wire, ws, res, options)
    good = wm.read_result(res)
    image, want_crc = wire[: good.wire_len].clone(), crc.clone()
    assert good.ok and good.wire_len < meta + n
    cap = good.wire_len                                              # (the tiles do not fit into it raw)
    wire.fill_(0xA5)
    t0 = time.time()
    with stalled(2):
        wm.wm_encode_opt(cur, chunk, None, crc, wire[:cap], ws, res, options)
        r = wm.read_result(res)
    assert r.status_name == "ERR_TIMEOUT" and wm.workspace_status(ws) == -10 and time.time() - t0 < 20
    assert bool((wire[cap:] == 0xA5).all()), "wrote past wire_cap"
    if tiles == 1:                                                   # the one tile is placed at the payload's start, raw
        assert r.wire_len == meta + 16384 and int(wire[64 + 16 * nc: 66 + 16 * nc].view(torch.int16)) == 512
    wm.wm_encode_opt(cur, chunk, None, crc, wire, ws, res, options)
    r = wm.read_result(res)
    assert r.ok and r.wire_len == good.wire_len and torch.equal(wire[: r.wire_len], image) and torch.equal(crc, want_crc)


@pytest.mark.parametrize("options", [0, wm.OPT_ENTROPY, wm.OPT_STRICT])
def test_decode_gives_up_when_the_copies_never_arrive(stalled, options):
    host, cur, chunk = _cache()
    n = cur.numel()
    nc = wm.num_chunks(n, chunk)
    ws, res = wm.new_workspace(n, chunk), wm.new_result()
    wire = torch.zeros(wm.wire_bound(n, chunk), dtype=torch.uint8, device="cuda")
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    wm.wm_encode_opt(cur, chunk, None, crc, wire, ws, res, options & wm.OPT_ENTROPY)
    r = wm.read_result(res)
    assert r.ok
    dst = torch.full((n,), 0x5A, dtype=torch.uint8, device="cuda")
    dst_crc = torch.full((nc,), 7, dtype=torch.int32, device="cuda")
    with stalled():
        wm.wm_decode_verify_opt(wire, r.wire_len, dst, chunk, dst_crc, ws, res, options)
        rd = wm.read_result(res)
    assert rd.status_name == "ERR_TIMEOUT" and wm.workspace_status(ws) == -10
    assert bool((dst_crc == 7).all()), "a checksum was installed after a timeout"
    if options & wm.OPT_STRICT:
        assert bool((dst == 0x5A).all()), "strict decode stored bytes before the verdict"
    wm.wm_decode_verify_opt(wire, r.wire_len, dst, chunk, dst_crc, ws, res, options)
    rd = wm.read_result(res)
    assert rd.ok and torch.equal(dst, cur) and torch.equal(dst_crc, crc)


def test_checksum_calls_fail_closed(stalled):
    host, cur, chunk = _cache()
    n = cur.numel()
    nc = wm.num_chunks(n, chunk)
    ws = wm.new_workspace(n, chunk)
    want = oracle.checksum(host.numpy(), chunk)
    for poly in (None, wm.POLY_ZLIB):
        crc = torch.full((nc,), 0x1234, dtype=torch.int32, device="cuda")
        with stalled():
            if poly is None:
                wm.wm_checksum(cur, chunk, crc, ws)
            else:
                wm.wm_checksum_poly(cur, chunk, poly, crc, ws)
            st = wm.workspace_status(ws)
        assert st == -10 and bool((crc == 0).all()), "digests of data that never arrived were delivered"
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    wm.wm_checksum(cur, chunk, crc, ws)
    assert wm.workspace_status(ws) == 0
    assert np.array_equal(crc.cpu().numpy().view(np.uint32), want)
    # the allocation-free call has the same channel (its built-in scratch: workspace None)
    with stalled():
        crc.fill_(5)
        wm.wm_checksum_noalloc(cur, chunk, crc)
        st = wm.workspace_status(None)
    assert st == -10 and bool((crc == 0).all())
    wm.wm_checksum_noalloc(cur, chunk, crc)
    assert wm.workspace_status(None) == 0
    assert np.array_equal(crc.cpu().numpy().view(np.uint32), want)


def test_dirty_diff_leaves_a_clean_status_even_on_a_dirty_workspace(stalled):
    host, cur, chunk = _cache()
    n = cur.numel()
    nc = wm.num_chunks(n, chunk)
    ws = wm.new_workspace(n, chunk)
    crc = torch.zeros(nc, dtype=torch.int32, device="cuda")
    with stalled():
        wm.wm_checksum(cur, chunk, crc, ws)
        assert wm.workspace_status(ws) == -10
    prev = cur.clone()
    prev[chunk * 3 + 17] ^= 1
    dirty = torch.zeros(nc, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    wm.wm_dirty_diff(cur, prev, chunk, dirty, None, cnt, ws)         # no waits inside: cannot time out
    assert wm.workspace_status(ws) == 0 and int(cnt.item()) == 1 and int(dirty[3].item()) == 1


@pytest.mark.parametrize("n,chunk", [(5 * 65536 + 777, 65536), (40 * 16384 + 31, 16384), (9, 16384), (3 << 20, 1 << 20),
                                     (-2, 16384), (-8, 16384), (-16, 16384)])
def test_xxh64_is_right_also_when_its_waits_run_out(stalled, n, chunk):
    """The call has no record to report a failure in: a wait that runs out costs time (the budget, not more), not the hash.
    -k: a chunk more than k for every SM, the last one short (a block of several chunks; of two chains, which share
    the word that says a wait has run out; blocks in two turns)."""
    turns = 1
    if n < 0:
        n_sm = torch.cuda.get_device_properties(0).multi_processor_count
        turns = 2 if n == -16 else 1
        n = -n * n_sm * chunk + 4097
    host = torch.randint(0, 256, (n,), dtype=torch.uint8, generator=torch.Generator().manual_seed(n))
    cur = host.cuda()
    out = torch.zeros(wm.num_chunks(n, chunk), dtype=torch.int64, device="cuda")
    want = oracle.checksum_xxh64(host.numpy(), chunk, seed=77).tolist()

    def timed():
        torch.cuda.synchronize()
        t0 = time.time()
        wm.wm_checksum_xxh64(cur, chunk, 77, out)
        torch.cuda.synchronize()
        return time.time() - t0
    timed()
    assert out.cpu().numpy().view(np.uint64).tolist() == want
    with stalled():
        out.fill_(5)
        spent = timed()
    assert out.cpu().numpy().view(np.uint64).tolist() == want
    assert spent < 1.0 * turns and (n < 32 or spent >= BUDGET_MS / 1000)     # (a chunk without a whole stripe waits for nothing)
    out.fill_(5)
    timed()
    assert out.cpu().numpy().view(np.uint64).tolist() == want


@pytest.mark.parametrize("tail", [0, 4097])
def test_checksum_of_a_large_cache_fails_closed(stalled, tail):
    """From 112 tiles per SM on a kernel of its own takes the cache, with a barrier per warp and eight waits per tile."""
    n, chunk = 113 * torch.cuda.get_device_properties(0).multi_processor_count * 16384 + tail, 1 << 20
    cur = torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda", generator=torch.Generator("cuda").manual_seed(tail))
    nc = wm.num_chunks(n, chunk)
    ws, crc = wm.new_workspace(n, chunk), torch.zeros(nc, dtype=torch.int32, device="cuda")

    def checksum(fill, poly=None):
        crc.fill_(fill)
        if poly is None:
            wm.wm_checksum(cur, chunk, crc, ws)
        else:
            wm.wm_checksum_poly(cur, chunk, poly, crc, ws)
        return wm.workspace_status(ws)
    assert checksum(0) == 0
    want = crc.clone()
    assert np.array_equal(want[-2:].cpu().numpy().view(np.uint32), oracle.checksum(cur[(nc - 2) * chunk:].cpu().numpy(), chunk))
    for poly in (None, wm.POLY_ZLIB):
        t0 = time.time()
        with stalled():
            assert checksum(0x1234, poly) == -10
        assert bool((crc == 0).all()) and time.time() - t0 < 20
        assert checksum(5) == 0 and torch.equal(crc, want)
