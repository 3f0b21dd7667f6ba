"""What the speed of this library is measured on: the mover's calls over the range its users have.

A case is one pass of a user's program on buffers it keeps (cache, wire, workspace, checksum
vectors):

  checksum   wm_checksum of a cache (the verification plane by itself)
  xxh64      wm_checksum_xxh64 of a cache
  encode     the source's half of a full move: fused checksum + encode
  decode     the destination's half: decode into the shadow buffer and verify
  move       both, one behind the other on one stream (source and destination share the GPU)
  step       one round of a live move: which chunks changed since the last snapshot, encode those,
             decode them into the destination's copy of the last snapshot

"data" is how the cache's values are distributed: "kv" keys with per-channel scales and outlier
channels and Gaussian values, "gauss" plain Gaussian, "bytes" incompressible, "llm" a text
model's append-only window that is filled in part and zero beyond.
"""
import math

import torch

from paper_2607_10389_b200 import binding as wm
from paper_2607_10389_b200 import inputs

KIB, MIB = 1 << 10, 1 << 20
ENGINE = 30 * 2 * 16 * 6800 * 128 * 2          # the engine cache: 1,671,168,000 bytes
LONG = 32 * 2 * 8 * 65536 * 128 * 2            # a long-context cache: 8 GiB
LLM = 24 * 2 * 8 * 16384 * 128 * 2             # a text model's whole window: 1.61 GB


def _case(path, nbytes, chunk, data="kv", entropy=False, zeros=False, strict=False, leaves=0, dirty=0.0, fill=1.0):
    return {"path": path, "nbytes": nbytes, "chunk": chunk, "data": data, "entropy": entropy, "zeros": zeros,
            "strict": strict, "leaves": leaves, "dirty": dirty, "fill": fill}


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)
    return [
        # the smallest call there is in use: a session's few control tensors, fingerprinted between two steps
        named("checksum_2m", "checksum", 2 * MIB, 64 * KIB, "gauss"),
        # fingerprint of the live cache against the manifest, without a move
        named("checksum_engine", "checksum", ENGINE, MIB),
        # the same with the 64-bit hash, where 32 bits are felt to be too few
        named("xxh64_engine", "xxh64", ENGINE, MIB),
        # a small session leaves: what counts is the length of the chain of launches
        named("encode_8m", "encode", 8 * MIB, 64 * KIB, "gauss"),
        # ... and arrives; its last tile is ragged, as a cache's that is no multiple of the tile
        named("decode_8m", "decode", 8 * MIB - 5000, 64 * KIB, "gauss"),
        # full move of the engine cache, the source's half and the destination's half
        named("encode_engine", "encode", ENGINE, MIB),
        named("decode_engine", "decode", ENGINE, MIB),
        # the same over a slow link: entropy-coded exponents
        named("move_engine_entropy", "move", ENGINE, MIB, entropy=True),
        # a round of live pre-copy: a generation step has rewritten three quarters of the chunks
        named("precopy_engine", "step", ENGINE, MIB, dirty=0.75),
        # a text model has appended tokens to its window; unused memory ships as table entries
        named("append_llm", "step", LLM, 64 * KIB, "llm", zeros=True, dirty=0.0682, fill=0.3172),
        # the cache as the engine holds it: 420 tensors of all sizes and 30 flags between them
        named("move_leaves", "move", inputs.PAPER_CACHE_BYTES, MIB, leaves=450),
        # a long-context cache moves
        named("move_long", "move", LONG, 4 * MIB),
    ]


CHUNKS = (16 * KIB, 64 * KIB, 64 * KIB, 240 * KIB, 256 * KIB, MIB, MIB, MIB, 4 * MIB)


def draw(rng):
    path = rng.choice(("checksum", "xxh64", "encode", "encode", "decode", "decode", "move", "move", "step", "step"))
    nbytes = int(2 ** rng.uniform(math.log2(256 * KIB), math.log2(3 << 30)))
    chunk = rng.choice(CHUNKS)
    if rng.random() < 0.5:
        nbytes &= ~255                           # whole rows of a head; otherwise any size at all
    if path in ("checksum", "xxh64"):
        return _case(path, nbytes, chunk, rng.choice(("kv", "gauss", "bytes")))
    if path == "step":
        if rng.random() < 0.4:
            fill = round(rng.uniform(0.25, 0.72), 4)
            return _case("step", nbytes, chunk, "llm", zeros=True, dirty=round(rng.uniform(0.001, 0.1), 4), fill=fill)
        return _case("step", nbytes, chunk, rng.choice(("kv", "gauss")), entropy=rng.random() < 0.2,
                     dirty=round(rng.uniform(0.02, 0.95), 3))
    data = rng.choice(("kv", "kv", "kv", "gauss", "bytes", "llm"))
    leaves = 15 * rng.randint(1, 40) if rng.random() < 0.3 and nbytes > 16 * MIB else 0
    return _case(path, nbytes, chunk, data, entropy=data != "bytes" and rng.random() < 0.25, zeros=data == "llm",
                 strict=path != "encode" and rng.random() < 0.25, leaves=leaves,
                 fill=round(rng.uniform(0.25, 0.72), 4) if data == "llm" else 1.0)


# ---------------------------------------------------------------- inputs

def _config(case, seed):
    """The cache recipe of at least case["nbytes"] bytes.  Small caches have fewer layers and heads."""
    n, data = case["nbytes"], case["data"]
    if data == "bytes":
        return inputs.CacheConfig("case", (), n, case["chunk"], seed, "bytes")
    layers, heads = (24, 8) if data == "llm" else (30, 16) if n >= 64 * MIB else (4, 8)
    dim = 64 if data == "gauss" else 128
    tokens = -(-n // (layers * 2 * heads * dim * 2))
    shape = (layers, 2, heads, tokens, dim)
    return inputs.CacheConfig("case", shape, layers * 2 * heads * tokens * dim * 2, case["chunk"], seed, data, case["fill"])


def _fit(t, n):
    """The first n bytes as a buffer of their own."""
    return t if t.numel() == n else t[:n].clone()


def _snapshots(case, seed):
    """(cache, previous snapshot) of a step."""
    cfg, n, chunk = _config(case, seed), case["nbytes"], case["chunk"]
    cache = inputs.make_cache(cfg, "cuda")
    if case["data"] == "llm":
        count = max(1, min(inputs.filled_tokens(cfg), round(case["dirty"] * cfg.shape[3])))
        prev, _ = inputs.before_append(cache, cfg, count)
        return _fit(cache, n), _fit(prev, n)
    prev = _fit(cache, n)
    cache = prev.clone()
    nc = -(-n // chunk)
    inputs.apply_step(cache, chunk, inputs.step_pattern(nc, min(30, nc), case["dirty"], seed), seed)
    return cache, prev


def _leaf_places(case):
    """(sizes, offsets) of the cache's tensors in the engine's pool, every one on a 256-byte boundary."""
    flags = case["leaves"] // 15
    sizes = inputs.paper_leaf_sizes(tensors=case["leaves"] - flags, flags=flags, total=case["nbytes"])
    offsets, at = [], 0
    for s in sizes:
        offsets.append(at)
        at += -(-s // 256) * 256
    return sizes, offsets, at


def _as_leaves(case, cache):
    """(pool, leaf table): the cache's bytes where the engine holds them; zeros when `cache` is None."""
    sizes, offsets, total = _leaf_places(case)
    pool = torch.zeros(total, dtype=torch.uint8, device="cuda")
    views, at = [], 0
    for s, o in zip(sizes, offsets):
        views.append(pool[o:o + s])
        if cache is not None:
            views[-1].copy_(cache[at:at + s])
        at += s
    return pool, wm.make_leaf_table(views)


def _u8(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def _u32(n):
    return torch.zeros(n, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    n, chunk, path = case["nbytes"], case["chunk"], case["path"]
    nc = wm.num_chunks(n, chunk)
    st = {"path": path, "n": n, "chunk": chunk, "table": None, "dst_table": None, "prev": None}
    if path == "step":
        st["cache"], st["prev"] = _snapshots(case, seed)
    else:
        st["cache"] = _fit(inputs.make_cache(_config(case, seed), "cuda"), n)
    if path == "xxh64":
        st["seed"], st["hash"] = seed & 0xFFFF, torch.zeros(nc, dtype=torch.int64, device="cuda")
        return st
    st["ws"], st["crc"] = wm.new_workspace(n, chunk), _u32(nc)
    if path == "checksum":
        return st

    # the codec's calls: buffers a sender and a receiver keep, and the image length the receiver is told
    st["enc_opt"] = (wm.OPT_ENTROPY if case["entropy"] else 0) | (wm.OPT_ZERO_TILES if case["zeros"] else 0)
    st["dec_opt"] = (wm.OPT_ENTROPY if case["entropy"] else 0) | (wm.OPT_STRICT if case["strict"] else 0)
    st["wire"], st["res"], st["dst_res"] = _u8(wm.wire_bound(n, chunk)), wm.new_result(), wm.new_result()
    st["dst_crc"] = _u32(nc)
    st["dirty"] = None
    if path == "step":
        st["dirty"], st["idx"], st["count"] = _u8(nc), _u32(nc), _u32(1)
        st["dst"] = st["prev"].clone()
        wm.wm_checksum(st["prev"], chunk, st["crc"], st["ws"])
        st["dst_crc"].copy_(st["crc"])
        _diff(st)
    else:
        if case["leaves"]:
            st["pool"], st["table"] = _as_leaves(case, st["cache"])
            st["dst"], st["dst_table"] = _as_leaves(case, None)
            st["cache"] = None
        else:
            st["dst"] = _u8(n)
    _encode(st)
    r = wm.read_result(st["res"])
    if not r.ok:
        raise RuntimeError(r.status_name)
    st["len"] = r.wire_len
    if path == "encode":
        st["dst"] = st["dst_table"] = None
    if path == "decode":
        st["cache"] = st["pool"] = st["table"] = None
    return st


# ---------------------------------------------------------------- one pass

def _diff(st):
    wm.wm_dirty_diff(st["cache"], st["prev"], st["chunk"], st["dirty"], st["idx"], st["count"], st["ws"])


def _encode(st):
    if st["enc_opt"]:
        wm.wm_encode_opt(st["cache"], st["chunk"], st["dirty"], st["crc"], st["wire"], st["ws"], st["res"], st["enc_opt"],
                         leaf_table=st["table"], nbytes=st["n"])
    elif st["table"] is not None:
        wm.wm_encode_leaves(st["table"], st["n"], st["chunk"], None, st["crc"], st["wire"], st["ws"], st["res"])
    else:
        wm.wm_encode(st["cache"], st["chunk"], st["dirty"], st["crc"], st["wire"], st["ws"], st["res"])


def _decode(st):
    if st["dec_opt"]:
        wm.wm_decode_verify_opt(st["wire"], st["len"], st["dst"] if st["dst_table"] is None else None, st["chunk"],
                                st["dst_crc"], st["ws"], st["dst_res"], st["dec_opt"], leaf_table=st["dst_table"],
                                nbytes=st["n"])
    elif st["dst_table"] is not None:
        wm.wm_decode_verify_leaves(st["wire"], st["len"], st["dst_table"], st["n"], st["chunk"], st["dst_crc"], st["ws"],
                                   st["dst_res"])
    else:
        wm.wm_decode_verify(st["wire"], st["len"], st["dst"], st["chunk"], st["dst_crc"], st["ws"], st["dst_res"])


def run(st):
    path = st["path"]
    if path == "checksum":
        wm.wm_checksum(st["cache"], st["chunk"], st["crc"], st["ws"])
        return st["crc"]
    if path == "xxh64":
        wm.wm_checksum_xxh64(st["cache"], st["chunk"], st["seed"], st["hash"])
        return st["hash"]
    out = {}
    if path == "step":
        _diff(st)
        out.update(dirty=st["dirty"], idx=st["idx"], count=st["count"])
    if path != "decode":
        _encode(st)
        out.update(wire=st["wire"], crc=st["crc"], res=st["res"])       # (zero behind the image: it was so before)
    if path != "encode":
        _decode(st)
        out.update(dst=st["dst"], dst_crc=st["dst_crc"], dst_res=st["dst_res"])
    return out


# ---------------------------------------------------------------- what a pass cannot do without

# Bytes of wire image per byte of cache, measured: (bit planes, entropy-coded exponents).
RATIO = {"kv": (0.757, 0.700), "gauss": (0.753, 0.687), "bytes": (1.0, 1.0), "llm": (0.757, 0.700)}


def work(case):
    """The cache read or written once on each side, the image written and read once; a step also
    reads both snapshots of a chunk until it has found a difference (a clean chunk: all of it).
    Checksums and codec are integer work: no floating-point operations are counted."""
    n, path = case["nbytes"], case["path"]
    if path in ("checksum", "xxh64"):
        return {"bytes": n, "flops": 0}
    ratio = RATIO[case["data"]][1 if case["entropy"] else 0]
    one = n * (1.0 + ratio)                      # one direction of a full move
    if case["data"] == "llm":
        one = n * (1.0 + ratio * case["fill"])
    if path == "step":
        share = case["dirty"]
        one = n * share * (1.0 + ratio)          # the dirty share is encoded and decoded
        return {"bytes": 2 * one + 2.0 * n * (1.0 - share), "flops": 0}
    return {"bytes": (2 if path == "move" else 1) * one, "flops": 0}


def tolerance(case):
    """Checksums, images and decoded bytes are what the format says they are, bit for bit."""
    return "exact"
