"""Performance cases of the paged tensor store, driven through its public Python calls.

Each case is one pass of a program that uses the store: what it put before the pass, the
buffers it owns and the batches it prepared once are made by ``prepare``; ``run`` makes the
calls. Calls go through ``put_prepared`` / ``get_prepared`` where a program's buffers stay the
same from call to call, as in a serving loop. Every output is a copy of stored bytes, or
their fp32 -> bf16 round-to-nearest-even cast, so every comparison is exact.

Kinds:

* ``handoff``   -- requests that hand text embeddings, pooled embeddings, latents and decoded
                   images from one model function to the next: put, get (latents with the
                   cast), free; on one stream or spread over several.
* ``pooled``    -- the same for the pooled embedding alone: one small tensor, where the cost of
                   a call is all there is.
* ``hit``       -- a window of one adapter (LoRA) set got from the adapter cache.
* ``miss``      -- a set that is not cached: put from pinned host memory, evicting the least
                   recent set, then a window of it got.
* ``weights``   -- whole transformer blocks of a cached model got in one call.
* ``small``     -- the biases and norm weights of a cached model's blocks got in one call.
* ``ragged``    -- objects of odd sizes packed back to back at any byte offset: put from one
                   packed buffer, got into another (every fourth with the cast), freed.
* ``compact``   -- weights that lie behind dead intermediates: put, the intermediates freed, the
                   pool compacted, the weights got, the pool grown back.
* ``pull``      -- a consumer's store pulls a request from a producer's, and gets it.
* ``noalloc``   -- one object gathered (with the cast) from a pool and its page list, without a
                   store.
"""
import math

import numpy as np
import torch

from paper_2607_26566_gb300 import Store, gather_noalloc, get_descs, put_descs

KiB, MiB = 1 << 10, 1 << 20
HIDDEN, MLP, HEAD = 3072, 12288, 128  # the 57-block DiT: 19 double blocks, then 38 single ones
N_DOUBLE, N_SINGLE = 19, 38


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest calls: one pooled embedding of one request (1.5 KiB)
        dict(name="pooled", kind="pooled", B=1, page_kib=2048),
        # eight single-image requests in flight on one stream, 22 MiB a call, fresh store
        dict(name="handoff_b1", kind="handoff", B=1, height=1024, width=1024, text_len=512, requests=8, streams=1,
             page_kib=2048, churn=False),
        # an odd resolution and prompt length, 64 KiB pages scattered by earlier use
        dict(name="handoff_b4_odd", kind="handoff", B=4, height=1216, width=840, text_len=333, requests=4, streams=1,
             page_kib=64, churn=True),
        # a busy server: sixteen B = 8 requests spread over four streams
        dict(name="handoff_b8_streams", kind="handoff", B=8, height=1024, width=1024, text_len=512, requests=16,
             streams=4, page_kib=2048, churn=True),
        # the adapter cache: a 256-object window of a rank-16 set, in 256 KiB pages
        dict(name="adapter_hit", kind="hit", rank=16, window=256, start=290, page_kib=256),
        # a rank-16 set (836 objects, 131 MB) reloaded from host, and its window
        dict(name="adapter_miss", kind="miss", rank=16, window=256, start=290, page_kib=256),
        # four double blocks restored to a consumer's buffers: the largest single call
        dict(name="weights", kind="weights", doubles=4, singles=0, page_kib=2048),
        # the 646 biases and norm weights that a quantised deployment keeps in bf16 beside
        # its packed matrices (256 B to 36 KiB each, 6 MB in all)
        dict(name="small_tensors", kind="small", doubles=19, singles=38, page_kib=64),
        # 40 objects of 1 KiB to 2 MiB at odd offsets
        dict(name="ragged", kind="ragged", objects=40, lo=1 * KiB, hi=2 * MiB, page_kib=64),
        # 1 GiB of weights moved when the pool shrinks
        dict(name="compact", kind="compact", mib=1024, hi=64 * MiB, page_kib=2048),
        # one B = 8 request pulled from a producer's store
        dict(name="pull", kind="pull", B=8, height=1024, width=1024, text_len=512, page_kib=2048),
        # sixteen images' fp32 latents (16 MiB) gathered without a store
        dict(name="noalloc", kind="noalloc", nbytes=16 * MiB, page_kib=2048),
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    """One more case of the same ranges: each kind, its sizes spread over their logarithm."""
    kind = rng.choice(["pooled", "handoff", "handoff", "handoff", "hit", "miss", "weights", "small", "ragged",
                       "compact", "pull", "noalloc"])
    pages = rng.choice([64, 256, 2048])
    if kind == "pooled":
        return dict(kind=kind, B=rng.randint(1, 64), page_kib=pages)
    if kind in ("handoff", "pull"):
        d = dict(kind=kind, B=rng.randint(1, 8), height=8 * rng.randint(32, 160), width=8 * rng.randint(32, 160),
                 text_len=rng.randint(20, 512), page_kib=pages)
        if kind == "handoff":
            d.update(requests=rng.randint(1, 12), streams=rng.randint(1, 4), churn=rng.random() < 0.5)
        return d
    if kind in ("hit", "miss"):
        window = _log(rng, 16, 400)
        return dict(kind=kind, rank=_log(rng, 4, 33), window=window, start=rng.randint(0, 836 - window), page_kib=256)
    if kind == "weights":
        return dict(kind=kind, doubles=rng.randint(0, 3), singles=rng.randint(1, 3), page_kib=rng.choice([256, 2048]))
    if kind == "small":
        return dict(kind=kind, doubles=rng.randint(1, 19), singles=rng.randint(0, 38), page_kib=rng.choice([64, 256]))
    if kind == "ragged":
        return dict(kind=kind, objects=_log(rng, 4, 400), lo=1 * KiB, hi=_log(rng, 16 * KiB, 4 * MiB), page_kib=pages)
    if kind == "compact":
        return dict(kind=kind, mib=_log(rng, 48, 1024), hi=_log(rng, 1 * MiB, 64 * MiB), page_kib=rng.choice([256, 2048]))
    return dict(kind=kind, nbytes=4 * _log(rng, 4 * KiB, 128 * MiB), page_kib=pages)


# ------------------------------------------------------------------ shapes
def _request(c):
    """(name, dtype, shape, cast) of one request's tensors."""
    lat = (c["B"], 16, c["height"] // 8, c["width"] // 8)
    return [("text", torch.bfloat16, (c["B"], c["text_len"], 4096), 0),
            ("pooled", torch.bfloat16, (c["B"], 768), 0),
            ("latents", torch.float32, lat, 1),
            ("image", torch.float16, (c["B"], 3, c["height"], c["width"]), 0)]


def _adapter_set(rank):
    """Bytes of a set's 836 objects: A [r, in] and B [out, r], bf16, of 418 projections."""
    h, m = HIDDEN, MLP
    proj = [(h, h)] * 4 + [(h, m), (m, h)]
    proj = proj * (2 * N_DOUBLE) + ([(h, h)] * 3 + [(h, m), (h + m, h)]) * N_SINGLE
    return [2 * rank * n for p in proj for n in p]


def _block_tensors(c):
    """Elements of each tensor (bf16) of the case's blocks, in checkpoint order."""
    h, m = HIDDEN, MLP
    double = 2 * ([h * h, h] * 4 + [m * h, m, h * m, h, 6 * h * h, 6 * h, HEAD, HEAD])
    single = [h * h, h] * 3 + [m * h, m, h * (h + m), h, 3 * h * h, 3 * h, HEAD, HEAD]
    sizes = double * c["doubles"] + single * c["singles"]
    return [n for n in sizes if n < h * h] if c["kind"] == "small" else sizes


def _log_sizes(g, n, lo, hi):
    return np.floor(np.exp(g.uniform(math.log(lo), math.log(hi), n))).astype(np.int64)


def _ragged(c):
    """(bytes, cast) of each packed object; sizes belong to the case, contents to the seed."""
    g = np.random.default_rng(c["objects"])
    n = _log_sizes(g, c["objects"], c["lo"], c["hi"])
    cast = np.arange(len(n)) % 4 == 3
    n[cast] &= ~3
    return n, cast.astype(np.uint32)


def _compact_sizes(c):
    """Object bytes of the compacted weights, c["mib"] MiB in all."""
    g, left, out = np.random.default_rng(c["mib"]), c["mib"] * MiB, []
    while left > 0:
        out.append(int(min(left, _log_sizes(g, 1, 4 * KiB, c["hi"])[0])))
        left -= out[-1]
    return np.array(out, np.int64)


def _pages(nbytes, page):
    return int(sum(-(-int(n) // page) for n in nbytes))


def _offsets(sizes, align=1):
    """Start of each object in one buffer, `align`-aligned, and the buffer's size."""
    ends = np.cumsum([-(-int(n) // align) * align for n in sizes])
    return np.concatenate([[0], ends[:-1]]).astype(np.uint64), int(ends[-1])


# ------------------------------------------------------------------ work, tolerance
def work(case):
    """Bytes that each call of a pass reads once and writes once."""
    c, k = case, case["kind"]
    if k == "pooled":
        n = 4 * 1536 * c["B"]
    elif k in ("handoff", "pull"):
        spec = _request(c)
        full = sum(math.prod(s) * t.itemsize for _, t, s, _ in spec)
        got = full - sum(math.prod(s) * 2 for _, _, s, cast in spec if cast)
        n = (2 * full + full + got) * c.get("requests", 1)
    elif k in ("hit", "miss"):
        sizes = _adapter_set(c["rank"])
        n = 2 * sum(sizes[c["start"]:c["start"] + c["window"]]) + (2 * sum(sizes) if k == "miss" else 0)
    elif k in ("weights", "small"):
        n = 2 * 2 * sum(_block_tensors(c))
    elif k == "ragged":
        sizes, cast = _ragged(c)
        n = 4 * int(sizes.sum()) - int(sizes[cast == 1].sum()) // 2
    elif k == "compact":
        n = 6 * int(_compact_sizes(c).sum())
    else:
        n = c["nbytes"] * 3 // 2
    return {"bytes": float(n), "flops": 0.0}


def tolerance(case):
    # copies, and a cast whose rounding is fixed: the same bits from every implementation
    return "exact"


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _tensor(g, dtype, shape):
    """bf16 and fp32: N(0, 1), as embeddings and latents; fp16: U[-1, 1], as decoded images."""
    x = torch.empty(shape, dtype=dtype, device="cuda")
    return x.uniform_(-1, 1, generator=g) if dtype == torch.float16 else x.normal_(0, 1, generator=g)


def _bytes(g, n):
    """n bytes of bf16 weights N(0, 0.02)."""
    return torch.empty(-(-n // 2), dtype=torch.bfloat16, device="cuda").normal_(0, 0.02, generator=g).view(torch.uint8)[:n]


def _store(n_pages, page, **kw):
    return Store(torch.empty(n_pages * page, dtype=torch.uint8, device="cuda"), page, **kw)


def _ok(store, status):
    if status:
        store.check(status)


def _churn(store, n_pages, page, seed):
    """Earlier use: the whole pool taken by objects of 1 to 8 pages and freed in another order."""
    g, sizes, left = np.random.default_rng(seed), [], n_pages
    while left:
        sizes.append(min(left, int(g.integers(1, 9))))
        left -= sizes[-1]
    st, ids = store.put_batch(put_descs(np.zeros(len(sizes), np.uint64), nbytes=np.array(sizes) * page))
    _ok(store, st)
    _ok(store, store.free(g.permutation(ids)))


def _stream():
    return int(torch.cuda.current_stream().cuda_stream)


def _put_all(store, sizes, g, offs, total, **kw):
    """Stores objects of one packed buffer of weights; their ids."""
    src = _bytes(g, total)
    st, ids = store.put_batch(put_descs(src.data_ptr() + offs, nbytes=sizes, **kw))
    _ok(store, st)
    torch.cuda.synchronize()  # src goes back to the allocator
    return ids


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    return {"case": case, **_PREPARE[case["kind"]](case, seed)}


def _prepare_handoff(c, seed):
    g, page = _gen(seed), c["page_kib"] * KiB
    spec = _request(c)
    R = c["requests"]
    n_pages = R * _pages([math.prod(s) * t.itemsize for _, t, s, _ in spec], page) + 8
    store = _store(n_pages, page)
    if c["churn"]:
        _churn(store, n_pages, page, seed)
    src = [_tensor(g, t, (R, *s)) for _, t, s, _ in spec]
    out = [torch.zeros((R, *s), dtype=torch.bfloat16 if cast else t, device="cuda") for _, t, s, cast in spec]
    casts = [cast for *_, cast in spec]
    puts = [store.prepare_put(put_descs([x[r] for x in src])) for r in range(R)]
    gets = [store.prepare_get(get_descs(np.zeros(len(spec), np.uint64), [x[r] for x in out], cast=casts))
            for r in range(R)]
    streams = [torch.cuda.Stream() for _ in range(c["streams"])] if c["streams"] > 1 else []
    on = [int(streams[r % len(streams)].cuda_stream) if streams else _stream() for r in range(R)]
    return dict(store=store, src=src, out=out, puts=puts, gets=gets, streams=streams, on=on)


def _prepare_pooled(c, seed):
    store = _store(64, c["page_kib"] * KiB)
    src = _tensor(_gen(seed), torch.bfloat16, (c["B"], 768))
    out = torch.zeros_like(src)
    return dict(store=store, src=[src], out=[out], puts=[store.prepare_put(put_descs([src]))],
                gets=[store.prepare_get(get_descs(np.zeros(1, np.uint64), [out]))], on=[_stream()])


def _window(c, sizes):
    return slice(c["start"], c["start"] + c["window"])


def _prepare_hit(c, seed):
    g, page, sizes = _gen(seed), c["page_kib"] * KiB, _adapter_set(c["rank"])
    n_pages = _pages(sizes, page)
    store = _store(n_pages + 64, page)
    _churn(store, n_pages + 64, page, seed)
    offs, total = _offsets(sizes, 256)
    ids = _put_all(store, sizes, g, offs, total, group=1, order=np.arange(len(sizes)), evictable=1)
    w = _window(c, sizes)
    at, n = _offsets(sizes[w], 256)
    out = torch.zeros(n // 2, dtype=torch.bfloat16, device="cuda")
    get = store.prepare_get(get_descs(ids[w], out.data_ptr() + at, dst_bytes=sizes[w]))
    return dict(store=store, out=out, get=get, ids=np.ascontiguousarray(ids[w]), on=_stream())


def _prepare_miss(c, seed):
    g, page, sizes = _gen(seed), c["page_kib"] * KiB, _adapter_set(c["rank"])
    store = _store(2 * _pages(sizes, page) + 64, page)  # two sets fit: each reload evicts the older
    offs, total = _offsets(sizes, 256)
    host = torch.empty(total, dtype=torch.uint8, pin_memory=True)
    host.copy_(_bytes(g, total))
    w = _window(c, sizes)
    at, n = _offsets(sizes[w], 256)
    out = torch.zeros(n // 2, dtype=torch.bfloat16, device="cuda")
    put = store.prepare_put(put_descs(host.data_ptr() + offs, nbytes=sizes, src_is_host=1, order=np.arange(len(sizes)),
                                      evictable=1))
    get = store.prepare_get(get_descs(np.zeros(c["window"], np.uint64), out.data_ptr() + at, dst_bytes=sizes[w]))
    return dict(store=store, host=host, out=out, put=put, get=get, window=w, group=0, on=_stream())


def _prepare_weights(c, seed):
    g, page = _gen(seed), c["page_kib"] * KiB
    sizes = [2 * n for n in _block_tensors(c)]
    offs, total = _offsets(sizes, 256)
    n_pages = _pages(sizes, page) + 8
    store = _store(n_pages, page)
    _churn(store, n_pages, page, seed)
    ids = _put_all(store, sizes, g, offs, total, group=1, order=np.arange(len(sizes)), evictable=1)
    out = torch.zeros(total // 2, dtype=torch.bfloat16, device="cuda")
    get = store.prepare_get(get_descs(ids, out.data_ptr() + offs, dst_bytes=sizes))
    return dict(store=store, out=out, get=get, ids=ids, on=_stream())


def _prepare_ragged(c, seed):
    g, page = _gen(seed), c["page_kib"] * KiB
    sizes, cast = _ragged(c)
    n_pages = _pages(sizes, page) + 8
    store = _store(n_pages, page)
    _churn(store, n_pages, page, seed)
    # the packed buffers start one element past an aligned address, as behind a header
    offs, total = _offsets(sizes)
    src = torch.randint(0, 256, (total + 3,), dtype=torch.uint8, device="cuda", generator=g)
    got = np.where(cast == 1, sizes // 2, sizes)
    at = np.zeros(len(got), np.uint64)
    pos = 2
    for i, n in enumerate(got):  # a cast writes bf16: its place is even
        pos += pos & int(cast[i])
        at[i] = pos
        pos += int(n)
    for i in np.flatnonzero(cast):  # the objects that are cast hold fp32 numbers
        x = torch.empty(int(sizes[i]) // 4, dtype=torch.float32, device="cuda").normal_(0, 1, generator=g)
        o = 3 + int(offs[i])
        src[o:o + int(sizes[i])] = x.view(torch.uint8)
    out = torch.zeros(pos, dtype=torch.uint8, device="cuda")
    put = store.prepare_put(put_descs(src.data_ptr() + 3 + offs, nbytes=sizes))
    get = store.prepare_get(get_descs(np.zeros(len(sizes), np.uint64), out.data_ptr() + at, dst_bytes=got, cast=cast))
    return dict(store=store, src=[src], out=[out], puts=[put], gets=[get], on=[_stream()])


def _prepare_compact(c, seed):
    g, page = _gen(seed), c["page_kib"] * KiB
    sizes = _compact_sizes(c)
    offs, total = _offsets(sizes, 256)
    n = _pages(sizes, page)
    store = _store(2 * n, page)
    src = _bytes(g, total)
    out = torch.zeros(total // 2, dtype=torch.bfloat16, device="cuda")
    dead = store.prepare_put(put_descs(np.zeros(1, np.uint64), nbytes=n * page))
    put = store.prepare_put(put_descs(src.data_ptr() + offs, nbytes=sizes))
    get = store.prepare_get(get_descs(np.zeros(len(sizes), np.uint64), out.data_ptr() + offs, dst_bytes=sizes))
    return dict(store=store, src=src, out=out, dead=dead, put=put, get=get, small=n * page, full=2 * n * page,
                on=_stream())


def _prepare_pull(c, seed):
    g, page = _gen(seed), c["page_kib"] * KiB
    spec = _request(c)
    n_pages = _pages([math.prod(s) * t.itemsize for _, t, s, _ in spec], page) + 8
    producer, consumer = _store(n_pages, page), _store(n_pages, page)
    _churn(producer, n_pages, page, seed)
    _churn(consumer, n_pages, page, seed + 1)
    src = [_tensor(g, t, s) for _, t, s, _ in spec]
    st, ids = producer.put_batch(put_descs(src))
    _ok(producer, st)
    out = [torch.zeros(s, dtype=torch.bfloat16 if cast else t, device="cuda") for _, t, s, cast in spec]
    get = consumer.prepare_get(get_descs(np.zeros(len(spec), np.uint64), out, cast=[cast for *_, cast in spec]))
    torch.cuda.synchronize()  # src goes back to the allocator
    return dict(producer=producer, store=consumer, ids=ids, out=out, get=get, on=_stream())


def _prepare_noalloc(c, seed):
    g, page = _gen(seed), c["page_kib"] * KiB
    n = -(-c["nbytes"] // page)
    pages = np.random.default_rng(seed).permutation(2 * n)[:n].astype(np.uint32)
    pool = _tensor(g, torch.float32, (2 * n * page // 4,)).view(torch.uint8)
    out = torch.zeros(c["nbytes"] // 4, dtype=torch.bfloat16, device="cuda")
    return dict(pool=pool, page=page, pages=pages, out=out, on=_stream())


_PREPARE = dict(handoff=_prepare_handoff, pooled=_prepare_pooled, hit=_prepare_hit, miss=_prepare_miss,
                weights=_prepare_weights, small=_prepare_weights, ragged=_prepare_ragged, compact=_prepare_compact,
                pull=_prepare_pull, noalloc=_prepare_noalloc)


# ------------------------------------------------------------------ run
def run(state):
    return _RUN[state["case"]["kind"]](state)


def _run_handoff(s):
    store, on = s["store"], s["on"]
    for p, stream in zip(s["puts"], on):
        _ok(store, store.put_prepared(p, stream)[0])
    for p, q, stream in zip(s["puts"], s["gets"], on):
        _ok(store, store.get_prepared(q, p.out, stream))
    for p in s["puts"]:
        _ok(store, store.free(p.out))
    return s["out"]


def _run_get(s):
    _ok(s["store"], s["store"].get_prepared(s["get"], s["ids"], s["on"]))
    return s["out"]


def _run_miss(s):
    store = s["store"]
    s["group"] += 1
    s["put"].descs["group"] = s["group"]
    st, ids = store.put_prepared(s["put"], s["on"])
    _ok(store, st)
    _ok(store, store.get_prepared(s["get"], ids[s["window"]], s["on"]))
    return s["out"]


def _run_compact(s):
    store, on = s["store"], s["on"]
    st, dead = store.put_prepared(s["dead"], on)
    _ok(store, st)
    st, ids = store.put_prepared(s["put"], on)
    _ok(store, st)
    _ok(store, store.free(dead))
    _ok(store, store.compact(s["small"], on)[0])
    _ok(store, store.get_prepared(s["get"], ids, on))
    _ok(store, store.free(ids))
    _ok(store, store.compact(s["full"], on)[0])
    return s["out"]


def _run_pull(s):
    store = s["store"]
    st, ids, _ = store.pull(s["producer"], s["ids"], stream=s["on"])
    _ok(store, st)
    _ok(store, store.get_prepared(s["get"], ids, s["on"]))
    _ok(store, store.free(ids))
    return s["out"]


def _run_noalloc(s):
    c = s["case"]
    if gather_noalloc(s["pool"], s["page"], s["pages"], c["nbytes"], s["out"], cast=1, stream=s["on"]):
        raise RuntimeError("gather_noalloc failed")
    return s["out"]


_RUN = dict(handoff=_run_handoff, pooled=_run_handoff, hit=_run_get, miss=_run_miss, weights=_run_get, small=_run_get,
            ragged=_run_handoff, compact=_run_compact, pull=_run_pull, noalloc=_run_noalloc)


# ------------------------------------------------------------------ exact
def exact(case, seed):
    """The inputs of the casts in 64 bits, where `run` returns them as numbers; None for plain copies."""
    c = case
    if c["kind"] in ("handoff", "pull"):
        g, R = _gen(seed), c.get("requests")
        x = [_tensor(g, t, (R, *s) if R else s) for _, t, s, _ in _request(c)]
        return [None, None, x[2].double(), None]
    if c["kind"] == "noalloc":
        page = c["page_kib"] * KiB
        n = -(-c["nbytes"] // page)
        pages = np.random.default_rng(seed).permutation(2 * n)[:n]
        pool = _tensor(_gen(seed), torch.float32, (2 * n, page // 4))
        return pool[torch.from_numpy(pages).cuda()].reshape(-1)[:c["nbytes"] // 4].double()
    return None
