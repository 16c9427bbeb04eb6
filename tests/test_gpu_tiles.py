"""Tiled launches (marked gpu) at the sizes where a tile can go wrong: objects
that end around a 16 KiB tile, pages of one tile and larger, pages smaller
than a tile (only runs of them are tiled), scattered and consecutive pages,
with and without the cast; put, get, compaction and pull. Every byte against
the input, the casts against the oracle's round-to-nearest-even."""
import numpy as np
import pytest
import torch

from oracle.cast import f32_bits_to_bf16_bits
from paper_2607_26566_gb300 import Store, gather_noalloc, get_descs, put_descs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
TILE = 16384


@pytest.fixture(scope="module", autouse=True)
def _built(lib):
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    yield


def scatter(st, n_pages, P, seed):
    """Free pages in a shuffled order."""
    s, ids = st.put_batch(put_descs(np.zeros(n_pages, np.uint64), nbytes=np.full(n_pages, P)))
    assert s == 0
    assert st.free(np.random.default_rng(seed).permutation(ids)) == 0


@pytest.mark.parametrize("big", [24 << 20, 256 << 10])   # a launch of many tiles, and a small one
@pytest.mark.parametrize("P,policy", [(16384, 0), (65536, 0), (2 << 20, 0), (4096, 1)])
def test_objects_that_end_around_a_tile(P, policy, big):
    rng = np.random.default_rng(P + policy)
    sizes = [big + 4] + [k * TILE + d for k in (1, 3) for d in (-16, -4, 0, 4, 16, 36)] + [4, 2 * P, 2 * P + 12]
    casts = [0] + [k % 2 for k in range(len(sizes) - 1)]
    datas = [rng.integers(0, 256, n, dtype=np.uint8) for n in sizes]
    n_pages = 2 * (sum(-(-n // P) for n in sizes) + 8)
    st = Store(torch.zeros(n_pages * P, dtype=torch.uint8, device=DEV), P, alloc_policy=policy)
    if policy == 0:
        scatter(st, n_pages, P, 3)
    srcs = [torch.from_numpy(d).to(DEV) for d in datas]
    s, dead = st.put_batch(put_descs([0], nbytes=[(n_pages // 2) * P]))
    s, ids = st.put_batch(put_descs(srcs))
    assert s == 0, st.last_error()
    want = [f32_bits_to_bf16_bits(d.view(np.uint32)).view(np.uint8) if c else d for d, c in zip(datas, casts)]

    def check(store, which):
        outs = [torch.full((w.size + 32,), 0xCD, dtype=torch.uint8, device=DEV) for w in want]
        assert store.get_batch(get_descs(which, outs, dst_bytes=[w.size for w in want], cast=casts))[0] == 0
        torch.cuda.synchronize()
        for o, w, n in zip(outs, want, sizes):
            h = o.cpu().numpy()
            assert np.array_equal(h[:w.size], w), n
            assert (h[w.size:] == 0xCD).all(), n

    check(st, ids)
    cons = Store(torch.zeros(n_pages * P, dtype=torch.uint8, device=DEV), P)
    s, pulled, _ = cons.pull(st, ids)
    assert s == 0
    check(cons, pulled)
    assert st.free(dead) == 0
    s, moved = st.compact((n_pages // 2) * P)
    assert s == 0 and moved > 0
    check(st, ids)


@pytest.mark.parametrize("P", [256, 2048, 4096, 65536])
@pytest.mark.parametrize("mis", [0, 1, 8, 14, 15])
def test_warp_tiles_at_their_edges(P, mis):
    """Small launches (warp tiles of 4 KiB): objects that end around a 16-byte
    vector and around a tile, sources and destinations `mis` bytes past a
    16-byte boundary, scattered pages smaller and larger than a tile, casts
    and copies in one call; the bytes around every destination stay."""
    rng = np.random.default_rng(P + mis)
    sizes = [k + d for k in (16, 4096, 8192, 40960) for d in (-15, -4, -1, 0, 1, 4, 15)] + [4, 8, 300 * P // 256]
    casts = [int(n % 4 == 0 and mis % 2 == 0) for n in sizes]
    datas = [rng.integers(0, 256, n, dtype=np.uint8) for n in sizes]
    n_pages = sum(-(-n // P) for n in sizes) + 3
    st = Store(torch.zeros(n_pages * P, dtype=torch.uint8, device=DEV), P)
    scatter(st, n_pages, P, 5)
    bufs = [torch.zeros(mis + n, dtype=torch.uint8, device=DEV) for n in sizes]
    for b, d in zip(bufs, datas):
        b[mis:] = torch.from_numpy(d).to(DEV)
    s, ids = st.put_batch(put_descs([b.data_ptr() + mis for b in bufs], nbytes=sizes))
    assert s == 0, st.last_error()
    assert st.stats()["launches"] == 1  # any mix of alignments is one launch
    for cast in (casts, [0] * len(sizes)):
        want = [f32_bits_to_bf16_bits(d.view(np.uint32)).view(np.uint8) if c else d for d, c in zip(datas, cast)]
        outs = [torch.full((mis + w.size + 32,), 0xCD, dtype=torch.uint8, device=DEV) for w in want]
        assert st.get_batch(get_descs(ids, [o.data_ptr() + mis for o in outs], dst_bytes=[w.size for w in want],
                                      cast=cast))[0] == 0
        torch.cuda.synchronize()
        for o, w, n in zip(outs, want, sizes):
            h = o.cpu().numpy()
            assert np.array_equal(h[mis:mis + w.size], w), n
            assert (h[:mis] == 0xCD).all() and (h[mis + w.size:] == 0xCD).all(), n


def test_gather_without_a_store_overlapping_and_captured():
    """gather_noalloc on four streams at once (no shared scratch), and captured
    into a CUDA graph after a kernel and after a copy that write its pool:
    every byte as the input's."""
    P, n = 65536, 9 << 20
    pages = np.random.default_rng(2).permutation(400)[:n // P].astype(np.uint32)
    pool = torch.randint(0, 256, (400 * P,), dtype=torch.uint8, device=DEV)
    want = pool.view(400, P)[torch.from_numpy(pages.astype(np.int64)).to(DEV)].reshape(-1)
    outs = [torch.zeros(n + 8, dtype=torch.uint8, device=DEV) for _ in range(4)]
    streams = [torch.cuda.Stream() for _ in range(4)]
    torch.cuda.synchronize()
    for _ in range(8):
        for k, (o, s) in enumerate(zip(outs, streams)):
            assert gather_noalloc(pool, P, pages, n, o.data_ptr() + k, dst_bytes=n, stream=s) == 0
    torch.cuda.synchronize()
    for k, o in enumerate(outs):
        assert torch.equal(o[k:k + n], want)
    src = pool.clone()
    out_a, out_b = torch.zeros(n, dtype=torch.uint8, device=DEV), torch.zeros(n, dtype=torch.uint8, device=DEV)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pool.bitwise_xor_(255)
        assert gather_noalloc(pool, P, pages, n, out_a) == 0
        pool.copy_(src)
        assert gather_noalloc(pool, P, pages, n, out_b) == 0
    for _ in range(3):
        out_a.zero_()
        out_b.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out_a, want ^ 255) and torch.equal(out_b, want)


@pytest.mark.parametrize("P", [16384, 65536, 1 << 20])
@pytest.mark.parametrize("n", [(4 << 20) + 20, (16 << 20) - 16, (16 << 20) + 20, (20 << 20) - 16, (20 << 20) + 20,
                               (48 << 20) + 4])
def test_large_calls_on_two_streams_in_turn(P, n):
    """Calls whose launches are shaped to run beside other streams' (and the
    first, which is not), on both sides of the line between warp and CTA tiles,
    in scattered pages: copy and cast, byte for byte."""
    n_pages = -(-n // P)
    st = Store(torch.zeros(2 * n_pages * P, dtype=torch.uint8, device=DEV), P)
    scatter(st, 2 * n_pages, P, 7)
    f = torch.randn(n // 4, device=DEV)
    outs = [torch.zeros(n, dtype=torch.uint8, device=DEV), torch.zeros(n // 2, dtype=torch.uint8, device=DEV)]
    torch.cuda.synchronize()
    for s in 2 * (torch.cuda.Stream(), torch.cuda.Stream()):
        st_, ids = st.put_batch(put_descs([f]), stream=s)
        assert st_ == 0
        assert st.get_batch(get_descs([ids[0], ids[0]], outs, cast=[0, 1]), stream=s)[0] == 0
        torch.cuda.synchronize()
        assert torch.equal(outs[0], f.view(torch.uint8))
        assert torch.equal(outs[1].view(torch.bfloat16), f.to(torch.bfloat16))
        assert st.free(ids) == 0
        outs[0].zero_()
        outs[1].zero_()
        torch.cuda.synchronize()


@pytest.mark.parametrize("n_obj", [4, 5, 6, 300])
def test_launches_with_a_segment_table(n_obj):
    """Objects of many tiles, as many as bring a table of segments with the
    launch and one fewer: sizes from one tile to a hundred, so that entries of
    the table cover several segments and part of one; put and get (copy)."""
    P = 65536
    rng = np.random.default_rng(n_obj)
    sizes = np.exp(rng.uniform(np.log(16384), np.log(100 * 16384), n_obj)).astype(np.int64) & ~15
    sizes[0] += max(0, (5 << 20) - int(sizes.sum()))
    offs = np.concatenate([[0], np.cumsum(sizes)])
    n_pages = int(sum(-(-n // P) for n in sizes)) + 5
    st = Store(torch.zeros(n_pages * P, dtype=torch.uint8, device=DEV), P)
    scatter(st, n_pages, P, 9)
    src = torch.randint(0, 256, (int(offs[-1]),), dtype=torch.uint8, device=DEV)
    s, ids = st.put_batch(put_descs(src.data_ptr() + offs[:-1], nbytes=sizes))
    assert s == 0, st.last_error()
    out = torch.zeros_like(src)
    assert st.get_batch(get_descs(ids, out.data_ptr() + offs[:-1], dst_bytes=sizes))[0] == 0
    torch.cuda.synchronize()
    assert torch.equal(out, src)


@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("mis,tiles_per_sm", [(0, k) for k in range(2, 10)]
                         + [(2, k) for k in (1, 4, 5, 8, 9, 17, 31, 32, 33)])
def test_one_wave_launches(mis, tiles_per_sm, extra):
    """Launches of a whole number of tiles for every SM, one more and one fewer
    (the CTA's threads follow from it): aligned (CTA tiles: 1,024 threads for two
    an SM down to 256 for eight, more than one wave for nine) and not (warp
    tiles, one CTA an SM up to 32 warps): a put, a get and a get with the cast
    of one fp32 object."""
    sms = torch.cuda.get_device_properties(DEV).multi_processor_count
    tile = 4096 if mis else TILE
    n = (tiles_per_sm * sms + extra) * tile - 4 * (tiles_per_sm % 3)
    P = 2 << 20
    st = Store(torch.zeros((n // P + 2) * P, dtype=torch.uint8, device=DEV), P)
    f = torch.randn(n // 4, device=DEV)
    src = torch.zeros(n + 16, dtype=torch.uint8, device=DEV)
    src[mis:mis + n] = f.view(torch.uint8)
    s, ids = st.put_batch(put_descs([src.data_ptr() + mis], nbytes=[n]))
    assert s == 0, st.last_error()
    out, bf = torch.zeros(n + 16, dtype=torch.uint8, device=DEV), torch.zeros(n // 2 + 16, dtype=torch.uint8, device=DEV)
    assert st.get_batch(get_descs(ids, [out.data_ptr() + mis], dst_bytes=[n]))[0] == 0
    assert st.get_batch(get_descs(ids, [bf.data_ptr() + mis], dst_bytes=[n // 2], cast=1))[0] == 0
    torch.cuda.synchronize()
    assert torch.equal(out[mis:mis + n], f.view(torch.uint8))
    assert torch.equal(bf[mis:mis + n // 2].view(torch.bfloat16), f.to(torch.bfloat16))
    for o, m in ((out, n), (bf, n // 2)):
        assert not o[:mis].any() and not o[mis + m:].any()
