"""The short-row search kernel on fp16 rows of 96 and 128 elements, and its instantiations for batches that do not
fill the GPU, against the CPU oracle.  ``visited=VISITED_BITMAP`` takes it at any batch size."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# d = 93: a row of 96 elements of which three are padding; 3,300 queries are 23 per SM, 60 are one
@pytest.mark.parametrize("d,storage,copies", [(93, 1, 1), (96, 1, 55), (128, 1, 1), (128, 1, 55), (96, 0, 1), (96, 0, 55)])
def test_every_pool(libs, tmp_path, d, storage, copies):
    rng = np.random.default_rng(d + copies)
    n = 5000
    centers = rng.standard_normal((10, d))
    base = (centers[rng.integers(0, 10, n)] + 0.4 * rng.standard_normal((n, d))).astype(np.float32)
    attrs = rng.integers(0, n, n).astype(np.int32)
    path = str(tmp_path / "x.idx")
    libs.build_index_gpu(base, attrs, path, ef_c=48)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    if storage:
        gix.enable_f16()
        ix = oracle.rounded_to_f16(ix)
    q = (base[rng.integers(0, n, 60)] + 0.2 * rng.standard_normal((60, d))).astype(np.float32)
    a = np.sort(attrs)
    w = (n * 2.0 ** -rng.uniform(0, 6, 60)).astype(int)
    s = (rng.random(60) * (n - w)).astype(int)
    lo, hi = a[s], a[s + w - 1]
    dev = [torch.from_numpy(np.ascontiguousarray(np.tile(x, (copies,) + (1,) * (x.ndim - 1)))).cuda() for x in (q, lo, hi)]
    for ef, budget in ((16, 16), (32, 64), (33, 64), (64, 24), (65, 128), (128, 64), (129, 64), (192, 128), (193, 128),
                       (256, 64), (257, 64), (512, 32)):
        ref = oracle.search(ix, q, lo, hi, 10, ef, B=budget)
        p = libs.Params(budget=budget, storage=storage, visited=libs.VISITED_BITMAP)
        status = torch.zeros(60 * copies, dtype=torch.int32, device="cuda")
        ids, dists = gix.search(*dev, 10, ef, params=p, status=status)
        torch.cuda.synchronize()
        assert np.array_equal(ids.cpu().numpy(), np.tile(ref.ids, (copies, 1)))
        assert np.array_equal(dists.cpu().numpy().view(np.uint32), np.tile(ref.dists.view(np.uint32), (copies, 1)))
        assert np.array_equal(status.cpu().numpy().view(np.uint32), np.tile(ref.status, copies))
        if copies == 1:
            q1 = [x[:60] for x in dev]
            other = gix.search_static(*q1, 10, ef, params=libs.Params(budget=budget, storage=storage))
            assert torch.equal(other[0], ids) and torch.equal(other[1], dists)
    gix.close()


# rows of 32 and 64 elements, two of them with padding; pools and budgets on both sides of the instantiations
@pytest.mark.parametrize("d,storage", [(32, 0), (30, 1), (64, 0), (61, 0), (64, 1)])
def test_rows_of_32_and_64(libs, tmp_path, d, storage):
    rng = np.random.default_rng(d)
    n, nq = 4000, 50
    base = rng.standard_normal((n, d)).astype(np.float32)
    attrs = rng.integers(0, n, n).astype(np.int32)
    path = str(tmp_path / "x.idx")
    libs.build_index_gpu(base, attrs, path, ef_c=48)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    if storage:
        gix.enable_f16()
        ix = oracle.rounded_to_f16(ix)
    q = (base[rng.integers(0, n, nq)] + 0.2 * rng.standard_normal((nq, d))).astype(np.float32)
    a = np.sort(attrs)
    w = (n * 2.0 ** -rng.uniform(0, 6, nq)).astype(int)
    s = (rng.random(nq) * (n - w)).astype(int)
    lo, hi = a[s], a[s + w - 1]
    for ef, budget in ((16, 16), (33, 64), (65, 128), (128, 64), (192, 128), (256, 64), (512, 32)):
        ref = oracle.search(ix, q, lo, hi, 10, ef, B=budget)
        for copies in (1, 80):                                           # one query per SM, and 28
            dev = [torch.from_numpy(np.ascontiguousarray(np.tile(x, (copies,) + (1,) * (x.ndim - 1)))).cuda() for x in (q, lo, hi)]
            for visited, flags in ((libs.VISITED_BITMAP, 0), (libs.VISITED_AUTO, 8)):      # bitmap, hash table where there is one
                ids, dists = gix.search(*dev, 10, ef, params=libs.Params(budget=budget, storage=storage, visited=visited, debug_flags=flags))
                torch.cuda.synchronize()
                assert np.array_equal(ids.cpu().numpy(), np.tile(ref.ids, (copies, 1)))
                assert np.array_equal(dists.cpu().numpy().view(np.uint32), np.tile(ref.dists.view(np.uint32), (copies, 1)))
    gix.close()


def test_fp16_batch_without_room_for_visited_slabs(libs):
    """600 queries need 170 MB of slabs on this index; where they cannot be had, the form that needs none runs."""
    import ctypes
    n, d, nq = 2_000_000, 96, 600
    vec = (np.arange(n * d, dtype=np.int32) * 7919 % 1021).astype(np.float32).reshape(n, d)
    rank = np.arange(n, dtype=np.int32)
    enc = np.full((n, 4), 0xFFFFFFFF, dtype=np.uint32)
    enc[:, 0] = (np.arange(n, dtype=np.int64) * 31 + 7) % n
    shape = libs.IndexInfo(n=n, d=d, d_pad=d, H=1, m=4)
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)

    def load():
        h = ctypes.c_void_p()
        assert libs._lib.frog_index_from_host(ptr(rank), ptr(rank), ptr(vec), ptr(enc), ctypes.byref(shape), 0, ctypes.byref(h)) == 0
        gix = libs.Index(h)
        gix.enable_f16()
        return gix

    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randint(0, 1000, (nq, d), generator=g, device="cuda").float()
    lo = torch.randint(0, n // 2, (nq,), generator=g, device="cuda", dtype=torch.int32)
    hi = lo + n // 3
    prm = libs.Params(budget=64, storage=1)
    out = [torch.empty((nq, 10), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
    gix = load()
    want = [t.clone() for t in gix.search(q, lo, hi, 10, 64, params=prm)]
    torch.cuda.synchronize()
    gix.close()
    gix = load()
    torch.cuda.empty_cache()
    fill = [torch.empty(torch.cuda.mem_get_info()[0] - (120 << 20), dtype=torch.uint8, device="cuda")]
    try:
        gix.search(q, lo, hi, 10, 64, params=prm, out_ids=out[0], out_dists=out[1])
        torch.cuda.synchronize()
    finally:
        fill.clear()
        torch.cuda.empty_cache()
    assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
    gix.close()
