"""Workloads whose time matters to a user of the library, through its public
calls (paper_2607_14431_gb300.kvg, the binding of include/kvg.h).

A case is one pass of one of these jobs:

  restore       a serving slot swaps its context: release, digest-verified
                graft of a stored block, append of the new prompt rows, decode
                of one token over everything
  host_restore  the same with the block in pinned host memory: a chunked,
                verified graft on a second stream, the decode split into slot
                ranges that follow the chunks
  decode        decode attention of one token per sequence, one layer (how a
                model calls it, layer by layer) or all layers
  step          one serving step of a batch: one appended row per sequence,
                then decode; every STEPS steps the conversations start again
                from their stored prefixes
  graft         graft of one block into a released slot, at its own position
                (verified or plain) or re-based by delta
  graft_batch   a library of blocks grafted into many sequences in one call
  deposit       a computed context captured as a block with its digests
  append        prefill rows written into a released slot

Geometries are those of the repository's workloads (kvg_synth.py): the tiny
fixture, the 12B class and the 31B class, on slices of their layers, and other
page sizes.  K, V and q are N(0, 1) draws rounded to bf16, as everywhere in
this repository; fp8 caches use its per-tensor scales.
"""
from __future__ import annotations

import math

import torch

from paper_2607_14431_gb300 import kvg

# query heads, kv heads, head_dim, page size, RoPE base
MODELS = {
    "tiny": (4, 2, 64, 16, 1e4),
    "12b": (16, 8, 256, 64, 1e4),
    "31b": (32, 16, 128, 64, 1e6),
}
FP8_SCALE = 0.0625  # per-tensor K and V scale of the fp8 caches
STEPS = 64          # decode steps a conversation runs before it starts again
SLAB = 1 << 30      # a store grows by slabs of at least this size


def listed():
    return [
        # the smallest call: a 256-token block swapped into a slot, one new
        # row, one decoded token; latency and launches count
        {"name": "restore_tiny", "kind": "restore", "model": "tiny", "layers": 2, "block": 256, "fresh": 1},
        # the headline workload: an 8,192-token block restored into a 32,768-
        # token context of the 12B class, verified beside the append
        {"name": "restore_12b", "kind": "restore", "model": "12b", "layers": 48, "block": 8192, "fresh": 24576,
         "overlap": True},
        # a block from the deep store in host memory
        {"name": "host_restore_12b", "kind": "host_restore", "model": "12b", "layers": 48, "block": 1024,
         "fresh": 4096},
        # one layer's attention, as a model calls it: a short chat ...
        {"name": "decode_layer_2k", "kind": "decode", "model": "31b", "layers": 2, "layer": 1, "batch": 1,
         "len_lo": 2111, "len_hi": 2111},
        # ... and a full 32k window
        {"name": "decode_layer_32k", "kind": "decode", "model": "12b", "layers": 2, "layer": 1, "batch": 1,
         "len_lo": 32768, "len_hi": 32768},
        # long contexts, several users, all layers of a slice in one call
        {"name": "decode_31b_64k", "kind": "decode", "model": "31b", "layers": 4, "layer": -1, "batch": 8,
         "len_lo": 65536, "len_hi": 65536},
        # continuous batching over contexts of different lengths
        {"name": "step_12b_b32", "kind": "step", "model": "12b", "layers": 2, "batch": 32, "len_lo": 8192,
         "len_hi": 24576},
        # the same on an fp8 cache, sliding-window layers but every second one
        {"name": "step_fp8_b16", "kind": "step", "model": "31b", "layers": 4, "batch": 16, "len_lo": 1000,
         "len_hi": 12001, "fp8": True, "window": 1024, "every": 2},
        # a block re-based to another offset
        {"name": "relocate_31b", "kind": "graft", "model": "31b", "layers": 20, "block": 16384, "delta": 4096},
        # a library of blocks of different lengths, verified
        {"name": "graft_batch_12b", "kind": "graft_batch", "model": "12b", "layers": 4, "batch": 16, "per_seq": 2,
         "len_lo": 2048, "len_hi": 6144, "verify": True},
        # a chat turn's context captured for later
        {"name": "deposit_12b", "kind": "deposit", "model": "12b", "layers": 48, "block": 499},
        # a prompt's rows quantized into an fp8 cache
        {"name": "append_fp8_12b", "kind": "append", "model": "12b", "layers": 48, "fresh": 3001, "fp8": True},
    ]


def _size(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]; odd ones as often as even."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["restore", "host_restore", "decode", "decode", "step", "step", "graft", "graft_batch",
                       "deposit", "append"])
    model = rng.choice(["tiny", "12b", "31b", "31b", "12b"])
    hq, hkv, d, page, _ = MODELS[model]
    case = {"kind": kind, "model": model}
    if rng.random() < 0.2:
        case["page"] = rng.choice([16, 32, 48, 128])
    fp8 = model != "tiny" and kind != "graft" and rng.random() < 0.3
    if fp8:
        case["fp8"] = True
    case["layers"] = layers = _size(rng, 2, 8 if model == "tiny" else 32)
    token = layers * 2 * hkv * d * 2  # bytes of one token's rows
    most = min(16384, (4 << 30) // token)
    if kind in ("restore", "host_restore"):
        case["block"] = _size(rng, 100, min(most, (512 << 20) // token if kind == "host_restore" else most))
        case["fresh"] = _size(rng, 1, most)
        if kind == "restore":
            case["overlap"] = rng.random() < 0.5
            if case["overlap"]:  # the append must not share the block's last page
                page = case.get("page", page)
                case["block"] = max(1, case["block"] // page) * page
    elif kind in ("decode", "step"):
        case["batch"] = batch = _size(rng, 1, 48)
        hi = _size(rng, 40, max(41, min(32768, 1000 * case.get("page", page), (8 << 30) // (token * batch))))
        case["len_lo"], case["len_hi"] = max(1, int(hi * rng.uniform(0.2, 1.0))), hi
        if kind == "decode":
            case["layer"] = rng.choice([-1, layers - 1])
        if rng.random() < 0.3:
            case["window"], case["every"] = _size(rng, 64, 2048), rng.choice([2, 3, 6])
    elif kind == "graft":
        case["block"] = _size(rng, 100, most)
        case["verify"] = rng.random() < 0.5
        if rng.random() < 0.5:
            case["delta"] = _size(rng, 1, 100000)
            case["interleaved"] = rng.random() < 0.5
    elif kind == "graft_batch":
        case["batch"], case["per_seq"] = _size(rng, 1, 24), rng.choice([1, 2, 3, 4])
        n = case["batch"] * case["per_seq"]
        hi = _size(rng, 64, max(65, min(6144, (4 << 30) // (token * n))))
        case["len_lo"], case["len_hi"] = max(1, hi // 3), hi
        case["verify"] = rng.random() < 0.6
        if not fp8 and rng.random() < 0.4:
            case["consecutive"] = True
    elif kind == "deposit":
        case["block"] = _size(rng, 100, min(most, (2 << 30) // token))
    else:
        case["fresh"] = _size(rng, 1, most)
    return case


# ------------------------------------------------------------- geometry --

def _geo(case):
    hq, hkv, d, page, theta = MODELS[case["model"]]
    return hq, hkv, d, int(case.get("page", page)), theta


def _dims(case):
    hq, hkv, d, page, theta = _geo(case)
    fp8 = bool(case.get("fp8"))
    return kvg.make_dims(case["layers"], hkv, d, page, theta,
                         kvg.KVG_ROPE_INTERLEAVED if case.get("interleaved") else kvg.KVG_ROPE_HALF,
                         kvg.KVG_KV_E4M3 if fp8 else kvg.KVG_KV_BF16, FP8_SCALE, FP8_SCALE)


def _lens(case, n):
    """Lengths of n sequences or blocks, spread evenly over [len_lo, len_hi] in a mixed order."""
    lo, hi = case["len_lo"], case["len_hi"]
    return [lo + (hi - lo) * ((i * 7919) % n) // max(1, n - 1) for i in range(n)]


def _windows(case):
    w, every = case.get("window", 0), case.get("every", 0)
    return [0 if not w or (l + 1) % every == 0 else w for l in range(case["layers"])]


def _layers_run(case):
    layer = case.get("layer", -1)
    return list(range(case["layers"])) if layer < 0 else [layer]


def _pages(case, n):
    page = _geo(case)[3]
    return (n + page - 1) // page


# --------------------------------------------------------------- inputs --

def _randn(seed, tag, shape):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + tag * 7919 + 17) & 0x7FFFFFFFFFFFFFFF)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)


def _rows(case, seed, tag, n):
    """K and V rows of n tokens, [layers][n][kv heads][head_dim]."""
    hq, hkv, d, _, _ = _geo(case)
    shape = (case["layers"], n, hkv, d)
    return _randn(seed, 2 * tag, shape), _randn(seed, 2 * tag + 1, shape)


def _queries(case, seed, batch):
    hq, hkv, d, _, _ = _geo(case)
    return _randn(seed, 999983, (len(_layers_run(case)), batch, hq, d))


def _arange(lo, n):
    return torch.arange(lo, lo + n, dtype=torch.int32, device="cuda")


class _Memory:
    """Device memory of a store or cache, as torch sees it; keeps its owner alive."""

    def __init__(self, owner, ptr, nbytes, typestr):
        self.owner = owner
        size = int(typestr[-1])
        self.__cuda_array_interface__ = {"shape": (int(nbytes) // size,), "typestr": typestr,
                                         "data": (int(ptr), False), "version": 3, "strides": None}


def _view(owner, ptr, nbytes, typestr):
    return torch.as_tensor(_Memory(owner, ptr, nbytes, typestr), device="cuda")


def _cache(case, pages, seqs, slots):
    """A cache whose pool starts as zeros (so that every byte of it is defined), and its state as tensors."""
    cache = kvg.Cache(_dims(case), pages, seqs, slots)
    v = cache.view
    if v.pool_bytes % 8 == 0:
        pool = _view(cache, v.pool, v.pool_bytes, "<i8")
    else:
        pool = _view(cache, v.pool, v.pool_bytes, "|u1")
    pool.zero_()
    tables = {"table": _view(cache, v.page_table, v.max_seqs * v.max_pages * 4, "<i4"),
              "fill": _view(cache, v.page_fill, v.max_seqs * v.max_pages * 4, "<i4"),
              "positions": _view(cache, v.positions, v.max_seqs * v.max_slots * 4, "<i4")}
    return cache, pool, tables


def _block_bytes(case, n):
    """A little more than the serialized size of a block of n tokens."""
    hq, hkv, d, page, _ = _geo(case)
    elem = 1 if case.get("fp8") else 2
    return (1 << 16) + 4 * n + case["layers"] * 2 * _pages(case, n) * (hkv * page * d * elem + 32)


def _library(case, seed, lens, residency=kvg.KVG_RESIDENCY_HBM):
    """A store with one block per length (block i: rows of tag i), written and deposited by another context."""
    total = sum(_block_bytes(case, n) for n in lens)
    store = kvg.Store(_dims(case), residency, total if len(lens) == 1 else 2 * total + 2 * SLAB)
    source = kvg.Cache(_dims(case), _pages(case, max(lens)), 1, max(lens))
    blocks = []
    for i, n in enumerate(lens):
        k, v = _rows(case, seed, i, n)
        p = _arange(0, n)
        kvg.kvg_cache_append(source.h, 0, k.data_ptr(), v.data_ptr(), p.data_ptr(), n)
        blocks.append(kvg.kvg_deposit(store.h, source.h, 0, 0, n))
        kvg.kvg_cache_release(source.h, 0)
        torch.cuda.current_stream().synchronize()
        del k, v, p
    torch.cuda.synchronize()
    source.close()
    return store, blocks


FRESH = 500000  # tag of the rows appended after a block
STEP = 600000   # tag of the rows of a serving step


def prepare(case, seed):
    kind = case["kind"]
    hq, hkv, d, page, _ = _geo(case)
    s = {"case": dict(case), "kind": kind, "hq": hq, "scale": 1.0 / math.sqrt(d),
         "stream": torch.cuda.current_stream().cuda_stream}
    if kind in ("restore", "host_restore"):
        nb, nf = case["block"], case["fresh"]
        host = kind == "host_restore"
        s["store"], blocks = _library(case, seed, [nb], kvg.KVG_RESIDENCY_PINNED_HOST if host
                                      else kvg.KVG_RESIDENCY_HBM)
        s["block"] = blocks[0]
        s["cache"], s["pool"], s["tables"] = _cache(case, _pages(case, nb + nf), 1, nb + nf)
        s["k"], s["v"] = _rows(case, seed, FRESH, nf)
        s["p"] = _arange(nb, nf)
        s["q"] = _queries(case, seed, 1)
        s["out"] = torch.empty_like(s["q"])
        s["side"] = torch.cuda.Stream()
        s["free"], s["done"] = torch.cuda.Event(), torch.cuda.Event()
        if host:
            # the part that is decoded while the block still crosses the link starts at a page boundary
            s["mid"] = nb // page * page
            s["slots"] = nb + nf
            s["state"] = torch.zeros(*s["q"].shape[:-1], d + 4, dtype=torch.float32, device="cuda")
            s["events"] = [torch.cuda.Event() for _ in range(16)]
            for e in s["events"]:
                e.record(s["side"])
    elif kind == "decode":
        lens = _lens(case, case["batch"])
        s["cache"], _, _ = _cache(case, sum(_pages(case, n) for n in lens), len(lens), max(lens))
        for i, n in enumerate(lens):
            k, v = _rows(case, seed, i, n)
            p = _arange(0, n)
            kvg.kvg_cache_append(s["cache"].h, i, k.data_ptr(), v.data_ptr(), p.data_ptr(), n)
            del k, v, p
        if case.get("window"):
            kvg.kvg_cache_set_layer_windows(s["cache"].h, _windows(case))
        s["seqs"] = list(range(len(lens)))
        s["q"] = _queries(case, seed, len(lens))
        s["out"] = torch.empty_like(s["q"])
    elif kind == "step":
        lens = _lens(case, case["batch"])
        s["store"], s["blocks"] = _library(case, seed, lens)
        s["cache"], s["pool"], s["tables"] = _cache(case, sum(_pages(case, n + STEPS) for n in lens), len(lens),
                                                    max(lens) + STEPS)
        if case.get("window"):
            kvg.kvg_cache_set_layer_windows(s["cache"].h, _windows(case))
        s["seqs"] = list(range(len(lens)))
        s["at"] = 0
        shape = (STEPS, case["layers"], len(lens), hkv, d)
        s["k"], s["v"] = _randn(seed, 2 * STEP, shape), _randn(seed, 2 * STEP + 1, shape)
        n = torch.tensor(lens, dtype=torch.int32, device="cuda")
        s["p"] = n[None] + torch.arange(STEPS, dtype=torch.int32, device="cuda")[:, None]
        s["rows"] = [(s["k"][t].data_ptr(), s["v"][t].data_ptr(), s["p"][t].data_ptr()) for t in range(STEPS)]
        s["q"] = _queries(case, seed, len(lens))
        s["out"] = torch.empty_like(s["q"])
        kvg.kvg_graft_batch(s["store"].h, s["blocks"], s["cache"].h, s["seqs"], 0, s["stream"])
    elif kind in ("graft", "graft_batch"):
        batch, per = case.get("batch", 1), case.get("per_seq", 1)
        lens = [case["block"]] if kind == "graft" else _lens(case, batch * per)
        s["store"], s["blocks"] = _library(case, seed, lens)
        s["seqs"] = [i // per for i in range(len(lens))]
        slots, deltas = _layout(case, lens, per)
        s["cache"], s["pool"], s["tables"] = _cache(case, sum(_pages(case, n) for n in lens), batch, slots)
        s["batch"], s["deltas"] = batch, deltas
        s["flags"] = kvg.KVG_GRAFT_VERIFY if case.get("verify") else 0
        if any(deltas):  # re-based keys are computed numbers
            s["pool"] = s["pool"].view(torch.bfloat16)
    elif kind == "deposit":
        n = case["block"]
        s["cache"], _, _ = _cache(case, _pages(case, n), 1, n)
        k, v = _rows(case, seed, 0, n)
        p = _arange(0, n)
        kvg.kvg_cache_append(s["cache"].h, 0, k.data_ptr(), v.data_ptr(), p.data_ptr(), n)
        s["dims"], s["n"], s["store"] = _dims(case), n, None
        size = _block_bytes(case, n)  # the store: four slabs
        s["capacity"], s["most"] = 4 * max(size, SLAB), 4 * max(1, min(16, SLAB // size))
    elif kind == "append":
        n = case["fresh"]
        s["cache"], s["pool"], s["tables"] = _cache(case, _pages(case, n), 1, n)
        s["k"], s["v"] = _rows(case, seed, 0, n)
        s["p"], s["n"] = _arange(0, n), n
    torch.cuda.synchronize()
    return s


def _layout(case, lens, per):
    """Slots the longest sequence needs (each block starts on a page) and each block's re-basing delta."""
    page = _geo(case)[3]
    slots, deltas = 0, []
    for i in range(0, len(lens), per):
        at = tokens = 0
        for n in lens[i:i + per]:
            at = (at + page - 1) // page * page + n
            deltas.append(tokens if case.get("consecutive") else case.get("delta", 0))
            tokens += n
        slots = max(slots, at)
    return slots, deltas


# ------------------------------------------------------------------ run --

def run(s):
    return _RUN[s["kind"]](s)


def _run_restore(s):
    c, main = s["cache"].h, s["stream"]
    kvg.kvg_cache_release(c, 0, main)
    if s["case"].get("overlap"):
        # the verified graft on a second stream, beside the append
        side = s["side"]
        s["free"].record()
        side.wait_event(s["free"])
        kvg.kvg_graft(s["store"].h, s["block"], c, 0, -1, 0, kvg.KVG_GRAFT_VERIFY, side.cuda_stream)
        s["done"].record(side)
        kvg.kvg_cache_append(c, 0, s["k"].data_ptr(), s["v"].data_ptr(), s["p"].data_ptr(), s["p"].numel(), main)
        torch.cuda.current_stream().wait_event(s["done"])
    else:
        kvg.kvg_graft(s["store"].h, s["block"], c, 0, -1, 0, kvg.KVG_GRAFT_VERIFY, main)
        kvg.kvg_cache_append(c, 0, s["k"].data_ptr(), s["v"].data_ptr(), s["p"].data_ptr(), s["p"].numel(), main)
    kvg.kvg_decode_attention(c, -1, [0], s["q"].data_ptr(), s["hq"], s["out"].data_ptr(), s["scale"], main)
    return {"out": s["out"], "pool": s["pool"], **s["tables"]}


def _run_host_restore(s):
    c, main, side = s["cache"].h, s["stream"], s["side"]
    stream = torch.cuda.current_stream()
    q, state = s["q"].data_ptr(), s["state"].data_ptr()
    kvg.kvg_cache_release(c, 0, main)
    s["free"].record()
    side.wait_event(s["free"])
    ends = kvg.kvg_graft_chunked(s["store"].h, s["block"], c, 0, [e.cuda_event for e in s["events"]],
                                 flags=kvg.KVG_GRAFT_VERIFY, stream=side.cuda_stream)
    s["done"].record(side)
    # a block that ends inside a page shares that page with the first fresh rows: they wait for its last chunk
    if s["mid"] != s["slots"] - s["p"].numel():
        stream.wait_event(s["events"][len(ends) - 1])
    kvg.kvg_cache_append(c, 0, s["k"].data_ptr(), s["v"].data_ptr(), s["p"].data_ptr(), s["p"].numel(), main)
    kvg.kvg_decode_attention_range(c, -1, [0], q, s["hq"], s["scale"], s["mid"], s["slots"], 0, state, main)
    lo = 0
    for j, hi in enumerate(ends):
        stream.wait_event(s["events"][j])
        hi = min(hi, s["mid"])
        if hi > lo:
            kvg.kvg_decode_attention_range(c, -1, [0], q, s["hq"], s["scale"], lo, hi, kvg.KVG_DECODE_MERGE, state,
                                           main)
        lo = hi
    stream.wait_event(s["done"])
    kvg.kvg_decode_state_finish(state, s["out"].numel() // s["out"].shape[-1], s["out"].shape[-1],
                                s["out"].data_ptr(), main)
    return {"out": s["out"], "state": s["state"], "pool": s["pool"], **s["tables"]}


def _run_decode(s):
    kvg.kvg_decode_attention(s["cache"].h, s["case"]["layer"], s["seqs"], s["q"].data_ptr(), s["hq"],
                             s["out"].data_ptr(), s["scale"], s["stream"])
    return s["out"]


def _run_step(s):
    c, main = s["cache"].h, s["stream"]
    if s["at"] == STEPS:  # the conversations are over: the next ones start from the stored prefixes
        for i in s["seqs"]:
            kvg.kvg_cache_release(c, i, main)
        kvg.kvg_graft_batch(s["store"].h, s["blocks"], c, s["seqs"], 0, main)
        s["at"] = 0
    k, v, p = s["rows"][s["at"]]
    s["at"] += 1
    kvg.kvg_cache_append_batch(c, s["seqs"], k, v, p, main)
    kvg.kvg_decode_attention(c, -1, s["seqs"], s["q"].data_ptr(), s["hq"], s["out"].data_ptr(), s["scale"], main)
    return {"out": s["out"], "pool": s["pool"], **s["tables"]}


def _run_graft(s):
    c, main = s["cache"].h, s["stream"]
    for i in range(s["batch"]):
        kvg.kvg_cache_release(c, i, main)
    if s["kind"] == "graft":
        kvg.kvg_graft(s["store"].h, s["blocks"][0], c, 0, -1, s["deltas"][0], s["flags"], main)
    else:
        kvg.kvg_graft_batch(s["store"].h, s["blocks"], c, s["seqs"], s["flags"], main,
                            deltas=s["deltas"] if any(s["deltas"]) else None)
    return {"pool": s["pool"], **s["tables"]}


def _run_deposit(s):
    if s["store"] is None or s["held"] == s["most"]:  # the store is full: a new one takes over
        if s["store"] is not None:
            s["store"].close()
        s["store"], s["held"] = kvg.Store(s["dims"], kvg.KVG_RESIDENCY_HBM, s["capacity"]), 0
    b = kvg.kvg_deposit(s["store"].h, s["cache"].h, 0, 0, s["n"], s["stream"])
    s["held"] += 1
    info = kvg.kvg_store_block_info(s["store"].h, b)  # the block's digest, which the program publishes
    return _view(s["store"], info.bytes, info.total_bytes, "|u1")


def _run_append(s):
    c, main = s["cache"].h, s["stream"]
    kvg.kvg_cache_release(c, 0, main)
    kvg.kvg_cache_append(c, 0, s["k"].data_ptr(), s["v"].data_ptr(), s["p"].data_ptr(), s["n"], main)
    return {"pool": s["pool"], **s["tables"]}


_RUN = {"restore": _run_restore, "host_restore": _run_host_restore, "decode": _run_decode, "step": _run_step,
        "graft": _run_graft, "graft_batch": _run_graft, "deposit": _run_deposit, "append": _run_append}


# ----------------------------------------------------------------- work --

def work(case):
    hq, hkv, d, page, _ = _geo(case)
    elem = 1 if case.get("fp8") else 2
    kind, layers = case["kind"], case["layers"]
    row = 2 * hkv * d  # K and V elements of one token in one layer

    def block(n):
        return layers * _pages(case, n) * page * row * elem

    def attention(lens):
        run, windows = _layers_run(case), _windows(case)
        rows = sum(min(n, windows[l]) if windows[l] else n for l in run for n in lens)
        return rows * row * elem + 2 * 2 * len(run) * len(lens) * hq * d, 4 * rows * hq * d

    def appended(rows):
        return rows * layers * row * (2 + elem)

    if kind in ("restore", "host_restore"):
        nb, nf = case["block"], case["fresh"]
        b, f = attention([nb + nf])
        return {"bytes": 2 * block(nb) + appended(nf) + b, "flops": f}
    if kind == "decode":
        b, f = attention(_lens(case, case["batch"]))
        return {"bytes": b, "flops": f}
    if kind == "step":
        b, f = attention([n + 1 for n in _lens(case, case["batch"])])
        return {"bytes": b + appended(case["batch"]), "flops": f}
    if kind == "graft":
        return {"bytes": 2 * block(case["block"]), "flops": 0}
    if kind == "graft_batch":
        return {"bytes": 2 * sum(block(n) for n in _lens(case, case["batch"] * case["per_seq"])), "flops": 0}
    if kind == "deposit":
        return {"bytes": 2 * block(case["block"]), "flops": 0}
    return {"bytes": appended(case["fresh"]), "flops": 0}


# ---------------------------------------------------------------- exact --

def _held(case, x):
    """A row as the cache holds it, in 64 bits."""
    if not case.get("fp8"):
        return x.double()
    return (x.float() * (1.0 / FP8_SCALE)).to(torch.float8_e4m3fn).double() * FP8_SCALE


def _attend(case, q, parts, out, at, windows):
    """Decode attention of one sequence in 64 bits: parts are its (K, V) rows in order; out[layer run][at]."""
    hq, hkv, d, _, _ = _geo(case)
    for i, l in enumerate(_layers_run(case)):
        k = torch.cat([_held(case, p[0][l]) for p in parts])
        v = torch.cat([_held(case, p[1][l]) for p in parts])
        if windows[l]:
            k, v = k[-windows[l]:], v[-windows[l]:]
        x = q[i, at].double().view(hkv, hq // hkv, d)
        w = torch.softmax(torch.einsum("hgd,nhd->hgn", x, k) / math.sqrt(d), dim=-1)
        out[i, at] = torch.einsum("hgn,nhd->hgd", w, v).reshape(hq, d)


def exact(case, seed):
    kind = case["kind"]
    windows = _windows(case)
    none = {"pool": None, "table": None, "fill": None, "positions": None}
    if kind in ("restore", "host_restore"):
        q = _queries(case, seed, 1)
        out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
        _attend(case, q, [_rows(case, seed, 0, case["block"]), _rows(case, seed, FRESH, case["fresh"])], out, 0,
                windows)
        return {"out": out, **none} if kind == "restore" else {"out": out, "state": None, **none}
    if kind in ("decode", "step"):
        lens = _lens(case, case["batch"])
        q = _queries(case, seed, len(lens))
        out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
        hq, hkv, d, _, _ = _geo(case)
        if kind == "step":
            shape = (STEPS, case["layers"], len(lens), hkv, d)
            k1, v1 = _randn(seed, 2 * STEP, shape)[0], _randn(seed, 2 * STEP + 1, shape)[0]
        for i, n in enumerate(lens):
            parts = [_rows(case, seed, i, n)]
            if kind == "step":
                parts.append((k1[:, i:i + 1], v1[:, i:i + 1]))
            _attend(case, q, parts, out, i, windows)
        return out if kind == "decode" else {"out": out, **none}
    if kind in ("graft", "graft_batch"):
        per = case.get("per_seq", 1)
        lens = [case["block"]] if kind == "graft" else _lens(case, case["batch"] * per)
        deltas = _layout(case, lens, per)[1]
        if not any(deltas):
            return None
        hq, hkv, d, page, theta = _geo(case)
        pool = torch.zeros(case["layers"], 2, sum(_pages(case, n) for n in lens), hkv, page, d, dtype=torch.float64,
                           device="cuda")
        w = theta ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device="cuda") / d)
        at = 0
        for i, (n, delta) in enumerate(zip(lens, deltas)):
            np_ = _pages(case, n)
            for kv, x in enumerate(_rows(case, seed, i, n)):
                y = torch.zeros(case["layers"], np_ * page, hkv, d, dtype=torch.float64, device="cuda")
                y[:, :n] = x.double()
                if kv == 0 and delta:
                    c, sn = torch.cos(delta * w), torch.sin(delta * w)
                    if case.get("interleaved"):
                        a, b = y[..., 0::2].clone(), y[..., 1::2].clone()
                        y[..., 0::2], y[..., 1::2] = a * c - b * sn, a * sn + b * c
                    else:
                        a, b = y[..., : d // 2].clone(), y[..., d // 2:].clone()
                        y[..., : d // 2], y[..., d // 2:] = a * c - b * sn, a * sn + b * c
                pool[:, kv, at:at + np_] = y.view(case["layers"], np_, page, hkv, d).transpose(2, 3)
            at += np_
        return {"pool": pool.view(-1), "table": None, "fill": None, "positions": None}
    return None


def tolerance(case):
    kind = case["kind"]
    if kind in ("append", "deposit"):
        return "exact"  # bytes
    if kind in ("graft", "graft_batch"):
        # bytes, but for re-based keys: an fp32 rotation rounded once to bf16
        # (0.0012 off 64 bits; one bf16 step is up to 2^-7 of a value)
        return {"rel": 0.005, "max": 0.01} if case.get("delta") or case.get("consecutive") else "exact"
    # attention: softmax weights rounded to 16 bits before the P.V product,
    # output rounded to bf16 (0.0017-0.0023 off 64 bits)
    return {"rel": 0.009, "max": 0.05}
