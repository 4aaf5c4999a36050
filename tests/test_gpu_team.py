"""The one-CTA-per-query search kernel (small batches) against the CPU oracle, at the edges of its pools, row
lengths, batch sizes and options.  ``visited=VISITED_AUTO`` takes it for these batch sizes."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _index(libs, tmp, n, d, seed, m=0, n_inv=-1):
    rng = np.random.default_rng(seed)
    centers = rng.standard_normal((12, d))
    base = (centers[rng.integers(0, 12, n)] + 0.4 * rng.standard_normal((n, d))).astype(np.float32)
    attrs = rng.integers(0, n // 2, n).astype(np.int32)                 # ties
    path = str(tmp / ("%d_%d.idx" % (n, d)))
    libs.build_index(base, attrs, path, m=m, n_inv=n_inv, ef_c=48)
    return base, attrs, path


def _queries(base, attrs, nq, seed):
    rng = np.random.default_rng(seed)
    n = len(attrs)
    q = (base[rng.integers(0, n, nq)] + 0.2 * rng.standard_normal((nq, base.shape[1]))).astype(np.float32)
    w = np.maximum(1, (n * 2.0 ** -rng.uniform(0, 7, nq)).astype(int))
    a = np.sort(attrs)
    s = (rng.random(nq) * (n - w + 1)).astype(int)
    lo, hi = a[s].copy(), a[s + w - 1].copy()
    if nq > 2:
        lo[1], hi[1] = hi[1] + 1, lo[1] - 1                              # empty
        lo[2], hi[2] = a[0], a[-1]                                       # everything
    return q, lo.astype(np.int32), hi.astype(np.int32)


def _run(libs, gix, q, lo, hi, k, ef, **kw):
    status = torch.zeros(len(lo), dtype=torch.int32, device="cuda")
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    ids, dists = gix.search(*dev, k, ef, params=libs.Params(**kw), status=status)
    torch.cuda.synchronize()
    assert gix.last_status() == 0
    return ids.cpu().numpy(), dists.cpu().numpy(), status.cpu().numpy().view(np.uint32)


# d: rows of 4 .. 3,072 bytes: below one 8-lane pass, ragged, one chunk, more than one, a ragged last chunk
@pytest.mark.parametrize("d,beams", [(1, (4, 33)), (30, (32, 65, 129)), (96, (1, 64, 128, 257)), (100, (31, 192)),
                                     (128, (48, 256, 512)), (130, (40, 100)), (300, (64,)), (768, (16, 200))])
def test_every_pool_and_row_length(libs, tmp_path, d, beams):
    base, attrs, path = _index(libs, tmp_path, 3000, d, d)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    q, lo, hi = _queries(base, attrs, 70, d + 1)
    for ef in beams:
        for budget in (16, 64, 128):
            got = _run(libs, gix, q, lo, hi, min(ef, 10), ef, budget=budget)
            ref = oracle.search(ix, q, lo, hi, min(ef, 10), ef, B=budget)
            assert np.array_equal(got[0], ref.ids) and np.array_equal(got[2], ref.status)
            assert np.array_equal(got[1].view(np.uint32), ref.dists.view(np.uint32))
    gix.close()


# batch sizes on both sides of the 8-warp form and of the resident grid, against the one-warp kernels
@pytest.mark.parametrize("d,storage", [(96, 0), (100, 0), (128, 1), (520, 0)])
def test_every_batch_size(libs, tmp_path, d, storage):
    base, attrs, path = _index(libs, tmp_path, 4000, d, d)
    gix = libs.Index.load(path)
    gix.enable_f16()
    q, lo, hi = _queries(base, attrs, 2400, 3)
    for nq in (1, 2, 63, 296, 297, 593, 1184, 1185, 2368, 2400):
        a = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], 10, 40, budget=32, storage=storage)
        b = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], 10, 40, budget=32, storage=storage, visited=libs.VISITED_BITMAP)
        for x, y in zip(a, b):
            assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
    gix.close()


# the lines between sixteen, eight and four warps per query and one, by batch size, budget and beam width
@pytest.mark.parametrize("d,storage", [(96, 0), (64, 1), (200, 0)])
def test_lines_between_the_forms(libs, tmp_path, d, storage):
    base, attrs, path = _index(libs, tmp_path, 4000, d, d)
    gix = libs.Index.load(path)
    gix.enable_f16()
    q, lo, hi = _queries(base, attrs, 900, 4)
    for budget, ef in ((47, 40), (48, 40), (128, 96), (128, 97), (64, 300)):
        for nq in (1, 148, 149, 297, 740, 741, 900):
            a = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], 10, ef, budget=budget, storage=storage)
            b = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], 10, ef, budget=budget, storage=storage, visited=libs.VISITED_BITMAP)
            for x, y in zip(a, b):
                assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
    gix.close()


# sixteen warps per query, which take their SM whole: every pool and row length
@pytest.mark.parametrize("d,storage", [(30, 0), (96, 1), (128, 0), (300, 0), (768, 1)])
def test_sixteen_warps(libs, tmp_path, d, storage):
    base, attrs, path = _index(libs, tmp_path, 3000, d, d)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    if storage:
        gix.enable_f16()
        ix = oracle.rounded_to_f16(ix)
    q, lo, hi = _queries(base, attrs, 37, d + 1)
    for ef in (1, 33, 65, 129, 257, 512):
        for budget, nq in ((48, 37), (128, 5)):
            got = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], min(ef, 10), ef, budget=budget, storage=storage)
            ref = oracle.search(ix, q[:nq], lo[:nq], hi[:nq], min(ef, 10), ef, B=budget)
            assert np.array_equal(got[0], ref.ids) and np.array_equal(got[2], ref.status)
            assert np.array_equal(got[1].view(np.uint32), ref.dists.view(np.uint32))
    gix.close()


def test_sixteen_warps_only_beside_nothing(libs, tmp_path, launches):
    """... so: a quarter of the SMs at most, and no other stream's search in flight."""
    base, attrs, path = _index(libs, tmp_path, 4000, 96, 1)
    quarter = torch.cuda.get_device_properties(0).multi_processor_count // 4
    steps = [dict(nq=nq, ef=40, budget=64, beside=beside) for nq, beside in
             ((1, 0), (quarter, 0), (quarter + 1, 0), (148, 0), (1, 1), (quarter, 1), (1, 0))]
    found = launches(path, *_queries(base, attrs, 6000, 4), steps)
    assert [[n for name, n in kernels if "team" in name] for kernels in found] == [[512], [512], [256], [256], [256], [256], [512]]


# four warps per query or one, on rows that the short-row kernel covers: storage, beam, budget, whether four
SHORT_ROWS = [(0, 96, 128, 0), (0, 97, 97, 1), (0, 160, 96, 0), (0, 256, 64, 0), (0, 257, 65, 1), (0, 384, 128, 1), (0, 385, 128, 0),
              (0, 512, 64, 0), (1, 160, 128, 0), (1, 257, 65, 1), (1, 257, 64, 0)]


def test_lines_on_short_rows(libs, tmp_path, launches):
    base, attrs, path = _index(libs, tmp_path, 4000, 96, 2)
    gix = libs.Index.load(path)
    gix.enable_f16()
    q, lo, hi = _queries(base, attrs, 740, 4)
    steps = []
    for storage, ef, budget, _ in SHORT_ROWS:
        for nq in (297, 740):
            steps.append(dict(nq=nq, ef=ef, budget=budget, storage=storage))
            a = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], 10, ef, budget=budget, storage=storage)
            b = _run(libs, gix, q[:nq], lo[:nq], hi[:nq], 10, ef, budget=budget, storage=storage, visited=libs.VISITED_BITMAP)
            for x, y in zip(a, b):
                assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
    gix.close()
    found = launches(path, q, lo, hi, steps)
    assert all(found)
    for step, kernels, team in zip(steps, found, np.repeat([x[3] for x in SHORT_ROWS], 2)):
        assert [n for name, n in kernels if "team" in name] == [128] * team, step


@pytest.mark.parametrize("kw,okw", [(dict(max_iters=1), dict(max_iters=1)), (dict(max_iters=7, budget=24), dict(max_iters=7, B=24)),
                                    (dict(epn=1), dict(epn=1)), (dict(epn=32, budget=1), dict(epn=32, B=1)),
                                    (dict(no_hotspot=1, budget=100), dict(no_hotspot=1, B=100)),
                                    (dict(exact_below=700, budget=32), dict(exact_below=700, B=32)),
                                    (dict(exact_below=4000), dict(exact_below=4000)), (dict(seed=12345), dict(seed=12345))])
def test_options(libs, tmp_path, kw, okw):
    base, attrs, path = _index(libs, tmp_path, 3000, 50, 9, m=20, n_inv=4)
    gix = libs.Index.load(path)
    q, lo, hi = _queries(base, attrs, 40, 5)
    ref = oracle.search(oracle.load_index(path), q, lo, hi, 8, 24, **okw)
    got = _run(libs, gix, q, lo, hi, 8, 24, **kw)
    assert np.array_equal(got[0], ref.ids) and np.array_equal(got[2], ref.status)
    assert np.array_equal(got[1].view(np.uint32), ref.dists.view(np.uint32))
    gix.close()


def test_non_finite_queries_and_rows(libs, tmp_path):
    """Distances that overflow or are not numbers are ordered by their bits, as in the other kernels."""
    base, attrs, path = _index(libs, tmp_path, 2000, 200, 4)
    gix = libs.Index.load(path)
    q, lo, hi = _queries(base, attrs, 24, 6)
    q[3, 5], q[4, 199], q[5, 0], q[6] = np.inf, np.nan, -np.inf, 2e19
    a = _run(libs, gix, q, lo, hi, 10, 48, budget=32)
    b = _run(libs, gix, q, lo, hi, 10, 48, budget=32, visited=libs.VISITED_BITMAP)
    for x, y in zip(a, b):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
    gix.close()
