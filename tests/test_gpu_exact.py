"""The exact filtered scan: grouped, split and one-CTA-per-query forms against the oracle's slab scan, at the
edges of its pieces, pools and row lengths.  From 17 queries on they are planned by a kernel of their own; which form
takes them then depends on their number, k and the size of the index, so that these sizes reach all of them."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _index(libs, tmp, n, d, seed):
    rng = np.random.default_rng(seed)
    base = rng.integers(0, 6, (n, d)).astype(np.float32)                # many equal distances: ties by id
    attrs = rng.integers(0, max(1, n // 3), n).astype(np.int32)
    path = str(tmp / ("e%d_%d.idx" % (n, d)))
    libs.build_index_gpu(base, attrs, path, m=4, ef_c=4, patience=1, n_inv=30)
    return base, attrs, path


def _queries(base, attrs, nq, seed, narrow):
    rng = np.random.default_rng(seed)
    n, d = base.shape
    q = (rng.integers(0, 60, (nq, d)) / 10).astype(np.float32)
    w = np.maximum(1, (n * 2.0 ** -rng.uniform(0, narrow, nq)).astype(int))
    a = np.sort(attrs)
    s = (rng.random(nq) * (n - w + 1)).astype(int)
    lo, hi = a[s].copy(), a[s + w - 1].copy()
    lo[0], hi[0] = a[0], a[-1]
    if nq > 1:
        lo[1], hi[1] = 5, 4                                              # empty
    if nq > 2:
        lo[2] = hi[2] = a[-1]
    return q, lo.astype(np.int32), hi.astype(np.int32)


def _check(gix, ix, q, lo, hi, k, graph=False):
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    if graph:
        out = (torch.empty((len(lo), k), dtype=torch.int32, device="cuda"), torch.empty((len(lo), k), device="cuda"))
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            gix.exact_search(*dev, k, out_ids=out[0], out_dists=out[1])
        g.replay()
    else:
        gix.exact_search(*dev, k)                                        # a first call may do without its scratch
        out = gix.exact_search(*dev, k)
    torch.cuda.synchronize()
    ids, dists = oracle.exact_slab(ix, q, lo, hi, k, mode=1)[:2]
    assert np.array_equal(out[0].cpu().numpy(), ids)
    assert np.array_equal(out[1].cpu().numpy().view(np.uint32), np.asarray(dists, np.float32).view(np.uint32))


@pytest.mark.parametrize("n,d", [(1, 3), (130, 16), (5000, 32), (20011, 50), (9000, 128), (3000, 300), (700, 6000)])
def test_matches_the_oracle(libs, tmp_path, n, d):
    base, attrs, path = _index(libs, tmp_path, n, d, n)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    for nq, narrow in ((1, 0), (6, 3), (16, 10), (17, 1), (200, 5), (203, 7)):
        q, lo, hi = _queries(base, attrs, nq, nq, narrow)
        for k in (1, 10, 33, 100) if n < 20000 else (10, 100):
            _check(gix, ix, q, lo, hi, k)
    q, lo, hi = _queries(base, attrs, 40 if n < 9000 else 210, 7, 4)
    for k in (64, 65, 129, 257, 512):
        _check(gix, ix, q, lo, hi, k)
        _check(gix, ix, q[:3], lo[:3], hi[:3], k)
    gix.close()


# Filtered scans (4,000 rows and more, many queries): rows that fill no tile of 128 or block of 32, row lengths on both
# sides of a pipeline stage, more queries than a tile has and than are listed at a time, k on both sides of what makes
# a slab wide, and an index too small for the bounds of all queries.
@pytest.mark.parametrize("n,d,nq", [(4000, 3, 129), (4127, 33, 260), (20011, 50, 100), (16001, 128, 2300), (5000, 260, 400), (70001, 8, 40)])
def test_filtered_scans(libs, tmp_path, n, d, nq):
    base, attrs, path = _index(libs, tmp_path, n, d, n)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    for narrow in (0, 4, 11) if nq < 2000 else (9,):
        q, lo, hi = _queries(base, attrs, nq, nq, narrow)
        for k in (1, 10, 40, 129, 512) if nq < 300 else (10, 100):
            _check(gix, ix, q, lo, hi, k)
    gix.close()


# slabs of fewer than 10 k rows are not filtered: without wider ones the form is for 100 (rows above 1 KB: 400) to 200 queries
@pytest.mark.parametrize("n,d,k,counts,filtered", [(5119, 20, 512, (100, 200, 201, 600), (1, 1, 0, 0)), (5120, 20, 512, (201, 600), (1, 1)),
                                                   (4000, 20, 401, (200, 201), (1, 0)), (4500, 260, 512, (200, 400), (0, 0))])
def test_long_lists_from_few_rows(libs, tmp_path, launches, n, d, k, counts, filtered):
    base, attrs, path = _index(libs, tmp_path, n, d, n)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    q, lo, hi = _queries(base, attrs, max(counts), 7, 6)
    for nq in counts:
        _check(gix, ix, q[:nq], lo[:nq], hi[:nq], k)
    gix.close()
    found = launches(path, q, lo, hi, [dict(nq=nq, k=k) for nq in counts])
    assert all(found)
    assert [any("filter_refine" in name for name, _ in kernels) for kernels in found] == [bool(x) for x in filtered]


@pytest.mark.parametrize("scale", [1.0, 1e-21, 3e17, 1e19])
def test_filtered_scans_of_extreme_values(libs, tmp_path, scale):
    """Products that underflow, overflow or are not numbers rule nothing out: same results, bit for bit, as the captured
    scan, which compares all rows."""
    rng = np.random.default_rng(8)
    n, d, nq = 9000, 40, 300
    base = (rng.standard_normal((n, d)) * scale).astype(np.float32)
    base[17, 3], base[18, 0], base[5000:5040, 1], base[77] = np.nan, np.inf, -np.inf, 3e38
    base[6000:6010] *= np.float32(1e6)
    attrs = rng.integers(0, n, n).astype(np.int32)
    path = str(tmp_path / "x.idx")
    libs.build_index_gpu(base, attrs, path, m=4, ef_c=4, patience=1, n_inv=30)
    gix = libs.Index.load(path)
    q = (rng.standard_normal((nq, d)) * scale).astype(np.float32)
    q[3, 5], q[4], q[5, 0], q[6], q[7] = np.inf, np.nan, -np.inf, 2e38, 0.0
    q[8] = base[6003]
    w = np.maximum(1, (n * 2.0 ** -rng.uniform(0, 5, nq)).astype(int))
    w[:9] = n
    s = (rng.random(nq) * (n - w + 1)).astype(int)
    a = np.sort(attrs)
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (q, a[s], a[s + w - 1])]
    for k in (1, 10, 100):
        want = [torch.empty((nq, k), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            gix.exact_search(*dev, k, out_ids=want[0], out_dists=want[1])
        graph.replay()
        for _ in range(2):
            got = gix.exact_search(*dev, k)
            torch.cuda.synchronize()
            assert torch.equal(got[0], want[0]) and torch.equal(got[1].view(torch.int32), want[1].view(torch.int32))
        graph.reset()
    gix.close()


@pytest.mark.parametrize("n,d,nq,k", [(100_000, 8, 9_001, 10), (20_011, 33, 20_003, 100), (400_003, 3, 2_001, 10)])
def test_filtered_scans_in_parts(libs, tmp_path, n, d, nq, k):
    """Batches over all rows that need several times the scratch there may be: bit for bit the captured scan, which
    compares all rows, and no more memory than the larger of 64 MB and half of the index."""
    rng = np.random.default_rng(n)
    base = rng.standard_normal((n, d)).astype(np.float32)
    path = str(tmp_path / "parts.idx")
    libs.build_index_gpu(base, rng.integers(0, n, n).astype(np.int32), path, m=4, ef_c=4, patience=1, n_inv=12)
    gix = libs.Index.load(path)
    q = torch.from_numpy(rng.standard_normal((nq, d)).astype(np.float32)).cuda()
    lo, hi = torch.zeros(nq, dtype=torch.int32, device="cuda"), torch.full((nq,), n, dtype=torch.int32, device="cuda")
    hi[::5] = n // 3
    hi[3::50] = 40
    out = [[torch.empty((nq, k), dtype=t, device="cuda") for t in (torch.int32, torch.float32)] for _ in range(2)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        gix.exact_search(q, lo, hi, k, out_ids=out[0][0], out_dists=out[0][1])
    graph.replay()
    gix.exact_search(q[:1], lo[:1], hi[:1], k)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(3):
        gix.exact_search(q, lo, hi, k, out_ids=out[1][0], out_dists=out[1][1])
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= max(64 << 20, gix.info.device_bytes // 2) + (4 << 20)
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1].view(torch.int32), out[1][1].view(torch.int32))
    graph.reset()
    gix.close()


def test_filtered_scans_of_norms_whose_sum_overflows(libs, tmp_path):
    """|q|^2 = 2e38: both norms and all distances are finite, the sum of the norms of q and a row like it is not."""
    rng = np.random.default_rng(2)
    n, d, nq = 6000, 40, 200
    q = rng.standard_normal((nq, d))
    q = (q * np.sqrt(2e38 / (q * q).sum(1, keepdims=True))).astype(np.float32)
    base = (rng.standard_normal((n, d)) * 5e17).astype(np.float32)
    for j, t in enumerate((1.0, 0.97, 0.5, 0.0, -0.3)):
        base[j:5 * nq:5] = np.float32(t) * q
    path = str(tmp_path / "x.idx")
    libs.build_index_gpu(base, rng.permutation(n).astype(np.int32), path, m=4, ef_c=4, patience=1, n_inv=30)
    ix, gix = oracle.load_index(path), libs.Index.load(path)
    lo, hi = np.zeros(nq, np.int32), np.full(nq, n, np.int32)
    hi[::7] = n // 2
    ids = gix.exact_search(*(torch.from_numpy(x).cuda() for x in (q, lo, hi)), 1)[0].cpu().numpy()[:, 0]
    all_rows = np.arange(nq) % 7 != 0
    assert np.array_equal(ids[all_rows], (5 * np.arange(nq))[all_rows])
    for k in (1, 3, 10):
        _check(gix, ix, q, lo, hi, k)
    gix.close()


def test_groups_with_gaps_streams_and_capture(libs, tmp_path):
    """Slabs that share no rows (a group's pieces jump the gaps), calls on two streams, and a captured call."""
    base, attrs, path = _index(libs, tmp_path, 30000, 24, 11)
    ix = oracle.load_index(path)
    gix = libs.Index.load(path)
    rng = np.random.default_rng(2)
    q, lo, hi = _queries(base, attrs, 1000, 3, 3)
    a = np.sort(attrs)
    s = rng.integers(0, 29000, 1000)
    lo[3:], hi[3:] = a[s][3:], a[s + rng.integers(0, 900, 1000)][3:]
    _check(gix, ix, q, lo, hi, 40)
    _check(gix, ix, q, lo, hi, 40, graph=True)
    _check(gix, ix, q[:5], lo[:5], hi[:5], 40, graph=True)
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    want = gix.exact_search(*dev, 40)
    streams = [torch.cuda.Stream() for _ in range(6)]
    torch.cuda.synchronize()
    got = []
    for i in range(24):
        with torch.cuda.stream(streams[i % 6]):
            n = (1000, 70, 7)[i % 3]
            got.append(gix.exact_search(*(x[:n] for x in dev), 40))
    torch.cuda.synchronize()
    for g in got:
        assert torch.equal(g[0], want[0][:len(g[0])]) and torch.equal(g[1], want[1][:len(g[0])])
    gix.close()


def test_reports_about_searches_are_left_alone(libs, tmp_path):
    """last_status and kernel_ms speak of the last SEARCH on a stream: exact scans, on the same stream or on
    another, with or without a search before them, change nothing about either."""
    base, attrs, path = _index(libs, tmp_path, 3000, 16, 5)
    q, lo, hi = _queries(base, attrs, 300, 6, 3)
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    a, b, c = (torch.cuda.Stream() for _ in range(3))
    torch.cuda.synchronize()

    def refused(call):
        with pytest.raises(libs.FrogError) as e:
            call()
        return e.value.code == 1

    gix = libs.Index.load(path)
    for n, k in ((3, 10), (100, 10), (300, 40)):
        gix.exact_search(*(x[:n] for x in dev), k, stream=a)
        a.synchronize()
        assert refused(lambda: gix.last_status(stream=a)) and refused(lambda: gix.kernel_ms(stream=a))
    gix.search(*dev, 10, 32, stream=b, params=libs.Params(debug_flags=16))
    b.synchronize()
    ms = gix.kernel_ms(stream=b)
    for n, k in ((3, 10), (100, 10), (300, 40)):
        for s in (b, c):
            gix.exact_search(*(x[:n] for x in dev), k, stream=s)
            s.synchronize()
            assert gix.last_status(stream=b) == 0 and gix.kernel_ms(stream=b) == ms
            assert refused(lambda: gix.last_status(stream=c)) and refused(lambda: gix.kernel_ms(stream=c))
    gix.close()


def test_the_per_thread_stream_is_another_stream_in_every_thread(libs, tmp_path):
    """Four threads, each on its own per-thread default stream (one handle, four streams): scans and searches of
    different batches do not share scratch."""
    import threading
    import types
    per_thread = types.SimpleNamespace(cuda_stream=2)
    base, attrs, path = _index(libs, tmp_path, 30000, 64, 9)
    gix = libs.Index.load(path)
    jobs = []
    for i, nq in enumerate((700, 90, 300, 1500)):
        dev = [torch.from_numpy(x).cuda() for x in _queries(base, attrs, nq, i, 5)]
        out = [torch.empty((nq, 20), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
        prm = libs.Params(visited=libs.VISITED_BITMAP)
        want = gix.exact_search(*dev, 20), gix.search(*dev, 20, 24, params=prm)
        jobs.append((dev, out, prm, want, []))
    torch.cuda.synchronize()
    gate = threading.Barrier(4)

    def work(dev, out, prm, want, bad):
        gate.wait()
        for i in range(60):
            if i % 2:
                gix.exact_search(*dev, 20, out_ids=out[0], out_dists=out[1], stream=per_thread)
            else:
                gix.search(*dev, 20, 24, out_ids=out[0], out_dists=out[1], stream=per_thread, params=prm)
            if i % 10 < 2:
                torch.cuda.synchronize()
                w = want[0 if i % 2 else 1]
                if not (torch.equal(out[0], w[0]) and torch.equal(out[1], w[1])):
                    bad.append(i)
        bad.append("done")

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [j[4] for j in jobs] == [["done"]] * 4
    # what is known about this thread's stream is not known about another's
    gix.search(*jobs[0][0], 20, 24, stream=per_thread)
    assert gix.last_status(stream=per_thread) == 0
    codes = []

    def ask():
        try:
            gix.last_status(stream=per_thread)
        except libs.FrogError as e:
            codes.append(e.code)

    t = threading.Thread(target=ask)
    t.start()
    t.join()
    assert codes == [1]
    gix.close()


def test_more_queries_than_a_planning_kernel_has_32_bit_threads(libs, tmp_path):
    """2^27 + 5 queries of one object each (one warp plans a query): as the same queries in small batches."""
    n, nq = 300_000, (1 << 27) + 5
    rng = np.random.default_rng(4)
    base = rng.standard_normal((n, 4)).astype(np.float32)
    path = str(tmp_path / "many.idx")
    libs.build_index_gpu(base, np.arange(n, dtype=np.int32), path, m=4, ef_c=4, patience=1, n_inv=12)
    gix = libs.Index.load(path)
    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randn(nq, 4, generator=g, device="cuda")
    lo = torch.randint(0, n, (nq,), generator=g, device="cuda", dtype=torch.int32)
    some = torch.cat([torch.randint(0, nq, (150,), generator=g, device="cuda"),
                      torch.tensor([0, 1, 1 << 26, (1 << 26) + 1, 1 << 27, nq - 1], device="cuda")])
    for call in (lambda *a: gix.exact_search(*a, 1), lambda *a: gix.search(*a, 1, 1)):
        ids, dists = call(q, lo, lo)
        want = call(q[some].contiguous(), lo[some].contiguous(), lo[some].contiguous())
        assert torch.equal(ids[:, 0], lo) and torch.equal(ids[some], want[0]) and torch.equal(dists[some], want[1])
    gix.close()


@pytest.mark.parametrize("n,d", [(300, 12), (9000, 33)])
def test_objects_of_several_vectors(libs, n, d):
    """An id that occurs several times, each time at another distance, is listed as often: in every form, and as in the
    scan of all rows."""
    import ctypes
    rng = np.random.default_rng(n)
    d_pad = (d + 3) // 4 * 4
    vec = np.zeros((n, d_pad), np.float32)
    vec[:, :d] = rng.standard_normal((n, d))
    attr, ids = np.arange(n, dtype=np.int32), rng.integers(0, n // 40, n).astype(np.int32)
    enc = np.full((n, 1, 4), 0xFFFFFFFF, np.uint32)
    shape = libs.IndexInfo(n=n, d=d, d_pad=d_pad, H=1, m=4)
    h = ctypes.c_void_p()
    assert libs._lib.frog_index_from_host(*[a.ctypes.data_as(ctypes.c_void_p) for a in (attr, ids, vec, enc)], ctypes.byref(shape), 0,
                                          ctypes.byref(h)) == 0
    gix = libs.Index(h)
    ix = oracle.OracleIndex(n=n, d=d, d_pad=d_pad, H=1, m=4, n_inv=0, ef_c=4, patience=1, beta=0.0, gamma=1.0, seed=0, sorted_attr=attr,
                            rank2id=ids, vectors=vec, enc=enc)
    q = rng.standard_normal((600, d)).astype(np.float32)
    lo = rng.integers(0, n // 2, 600).astype(np.int32)
    hi = (lo + rng.integers(0, n // 2, 600)).astype(np.int32)
    for nq in (1, 6, 30, 250, 600):
        for k in (10, 60, 300):
            _check(gix, ix, q[:nq], lo[:nq], hi[:nq], k)
    gix.close()


def test_scans_beside_another_threads_capture(libs, tmp_path):
    """A thread captures a graph; another one scans an index for the first time, which allocates.  The scan works
    and the capture is not spoilt."""
    import threading
    base, attrs, path = _index(libs, tmp_path, 20000, 40, 3)
    q, lo, hi = _queries(base, attrs, 400, 8, 5)
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    gix, side = libs.Index.load(path), torch.cuda.Stream()
    calls = ((400, 50), (100, 10), (5, 10), (400, 200))
    want = [[t.cpu() for t in gix.exact_search(*(x[:n] for x in dev), k)] for n, k in calls]
    gix.close()
    gix = libs.Index.load(path)
    parts = [[x[:n].contiguous() for x in dev] for n, _ in calls]
    out = [[torch.empty((n, k), dtype=t, device="cuda") for t in (torch.int32, torch.float32)] for n, k in calls]
    x, errors = torch.zeros(1000, device="cuda"), []
    torch.cuda.synchronize()

    def scan():
        try:
            for (n, k), p, o in zip(calls, parts, out):
                gix.exact_search(*p, k, out_ids=o[0], out_dists=o[1], stream=side)
        except libs.FrogError as e:
            errors.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x += 1
        t = threading.Thread(target=scan)
        t.start()
        t.join()
        x += 1
    graph.replay()
    torch.cuda.synchronize()
    assert not errors and float(x[0]) == 2.0
    for o, w in zip(out, want):
        assert torch.equal(o[0].cpu(), w[0]) and torch.equal(o[1].cpu(), w[1])
    gix.close()


def test_a_first_scan_of_common_size_allocates_nothing(libs, tmp_path):
    """The scratch of up to 2,048 queries with k up to 128 comes with the index, as far as half of its size."""
    base, attrs, path = _index(libs, tmp_path, 50000, 96, 3)
    ix = oracle.load_index(path)
    q, lo, hi = _queries(base, attrs, 2048, 8, 6)
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    for nq, k in ((1, 10), (16, 128), (200, 128), (500, 10), (2048, 10), (2048, 20)):
        gix = libs.Index.load(path)
        out = [torch.empty((nq, k), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
        part = [x[:nq] for x in dev]
        if nq == 1:                                         # the library's kernels are loaded
            gix.exact_search(*(x[:600] for x in dev), 100)
            gix.exact_search(*(x[:100] for x in dev), 100)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        gix.exact_search(*part, k, out_ids=out[0], out_dists=out[1])
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == before
        ids, _ = oracle.exact_slab(ix, q[:nq], lo[:nq], hi[:nq], k, mode=1)[:2]
        assert np.array_equal(out[0].cpu().numpy(), ids)
        gix.close()


@pytest.mark.parametrize("n,d,nq,k", [(5000, 128, 2000, 100), (8000, 8, 400, 512)])
def test_a_first_scan_of_a_small_index_allocates_nothing(libs, tmp_path, n, d, nq, k):
    """It needs more than came with the index, and does without whichever form it takes."""
    base, attrs, path = _index(libs, tmp_path, n, d, 5)
    ix = oracle.load_index(path)
    q, lo, hi = _queries(base, attrs, nq, 8, 6)
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    out = [torch.empty((nq, k), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
    ids, _ = oracle.exact_slab(ix, q, lo, hi, k, mode=1)[:2]
    for load in range(2):                                   # the first loads the library's kernels
        gix = libs.Index.load(path)
        free = []
        for call in range(3):
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
            out[0].zero_()
            gix.exact_search(*dev, k, out_ids=out[0], out_dists=out[1])
            assert np.array_equal(out[0].cpu().numpy(), ids)
        gix.close()
    assert free[1] == free[0]


@pytest.mark.parametrize("d", [57300, 57520])
def test_the_longest_rows_that_fit_one_query(libs, tmp_path, d):
    """Rows of 229,200 and 230,080 bytes: the scan without pieces needs 2,048 bytes of shared memory besides."""
    rng = np.random.default_rng(d)
    base = rng.integers(0, 3, (40, d)).astype(np.float32)
    path = str(tmp_path / "long.idx")
    libs.build_index(base, rng.integers(0, 20, 40).astype(np.int32), path, m=4, ef_c=4, n_inv=30)
    ix, gix = oracle.load_index(path), libs.Index.load(path)
    for nq in (3, 40):
        lo = rng.integers(0, 15, nq).astype(np.int32)
        _check(gix, ix, rng.integers(0, 3, (nq, d)).astype(np.float32), lo, lo + 5, 10)
    gix.close()


def test_two_threads_whose_calls_need_different_shared_memory(libs, tmp_path):
    """Long and short rows through the same kernels: what one thread allows a kernel, the other does not take back."""
    import threading
    work = []
    for d, n in ((3000, 300), (40, 2000)):
        rng = np.random.default_rng(d)
        base = rng.standard_normal((n, d)).astype(np.float32)
        path = str(tmp_path / ("sm%d.idx" % d))
        libs.build_index(base, np.arange(n, dtype=np.int32), path, m=4, ef_c=4, n_inv=30)
        gix = libs.Index.load(path)
        q = torch.from_numpy(base[:300]).cuda()
        lo, hi = torch.zeros(300, dtype=torch.int32, device="cuda"), torch.full((300,), n, dtype=torch.int32, device="cuda")
        calls = []
        for nq, k, beam in ((300, 400, 0), (300, 40, 0), (100, 400, 0), (8, 400, 0), (50, 10, 290)):
            a = (q[:nq], lo[:nq], hi[:nq], k) + ((beam,) if beam else ())
            kw = dict(out_ids=torch.empty((nq, k), dtype=torch.int32, device="cuda"), out_dists=torch.empty((nq, k), device="cuda"))
            want = [t.clone() for t in (gix.search if beam else gix.exact_search)(*a, **kw)]
            calls.append((gix.search if beam else gix.exact_search, a, dict(kw, stream=torch.cuda.Stream()), want))
        work.append((calls, []))
    torch.cuda.synchronize()
    gate = threading.Barrier(2)

    def run(calls, errors):
        gate.wait()
        try:
            for _ in range(300):
                for f, a, kw, want in calls:
                    f(*a, **kw)
            torch.cuda.synchronize()
            assert all(torch.equal(kw["out_ids"], w[0]) and torch.equal(kw["out_dists"], w[1]) for f, a, kw, w in calls)
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert [w[1] for w in work] == [[], []]


def test_more_streams_in_flight_than_scratch_sets(libs, tmp_path):
    """20 streams: the last of them scan without scratch, with the same results."""
    base, attrs, path = _index(libs, tmp_path, 60000, 64, 21)
    gix = libs.Index.load(path)
    q, lo, hi = _queries(base, attrs, 400, 3, 2)
    dev = [torch.from_numpy(x).cuda() for x in (q, lo, hi)]
    want = gix.exact_search(*dev, 50)
    streams = [torch.cuda.Stream() for _ in range(20)]
    torch.cuda.synchronize()
    got = []
    for i in range(60):
        n = (400, 60, 9)[i // 20]
        out = [torch.empty((n, 50), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
        got.append(out)
    torch.cuda.synchronize()
    for i, out in enumerate(got):
        gix.exact_search(*(x[:len(out[0])] for x in dev), 50, out_ids=out[0], out_dists=out[1], stream=streams[i % 20])
    torch.cuda.synchronize()
    for g in got:
        assert torch.equal(g[0], want[0][:len(g[0])]) and torch.equal(g[1], want[1][:len(g[0])])
    gix.close()
