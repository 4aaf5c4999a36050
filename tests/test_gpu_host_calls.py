"""Host-buffer searches: every mix of pinned and pageable buffers, on both sides of what the index's own page-locked buffer
holds, from two threads at once; the results are those of the device call."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_pinned_and_pageable_buffers(libs, tmp_path):
    rng = np.random.default_rng(3)
    n, d, nq, k = 5000, 96, 1200, 10
    base = rng.standard_normal((n, d)).astype(np.float32)
    attrs = rng.integers(0, n, n).astype(np.int32)
    path = str(tmp_path / "x.idx")
    libs.build_index_gpu(base, attrs, path, ef_c=32)
    gix = libs.Index.load(path)
    a = np.sort(attrs)
    w = np.maximum(1, (n * 2.0 ** -rng.uniform(0, 7, nq)).astype(int))
    s = (rng.random(nq) * (n - w + 1)).astype(int)
    host = [torch.from_numpy(np.ascontiguousarray(x)) for x in (base[:nq] + 0.1, a[s], a[s + w - 1])]
    want = [x.cpu() for x in gix.search(*(x.cuda() for x in host), k, 32)]

    def call(size, pinned, stream):
        src = [x[:size].contiguous().pin_memory() if p else x[:size].clone() for x, p in zip(host, pinned)]
        out = [torch.full((size, k), -7, dtype=t) for t in (torch.int32, torch.float32)]
        out = [x.pin_memory() if p else x for x, p in zip(out, pinned[3:])]
        gix.search_host(*src, k, 32, out_ids=out[0], out_dists=out[1], stream=stream)
        return torch.equal(out[0], want[0][:size]) and torch.equal(out[1].view(torch.int32), want[1][:size].view(torch.int32))

    # 610 queries and their results are 283 KB pageable, of which the queries are 234 KB
    for size in (1, 16, 610, 1200):
        for mask in range(32):
            assert call(size, [bool(mask >> i & 1) for i in range(5)], None), (size, mask)

    bad = []

    def work(seed):
        stream = torch.cuda.Stream()
        r = np.random.default_rng(seed)
        for _ in range(30):
            if not call(int(r.integers(1, 700)), list(r.random(5) < 0.4), stream):
                bad.append(seed)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    gix.close()


def _small(libs, tmp_path):
    rng = np.random.default_rng(5)
    n, d = 3000, 32
    base = rng.standard_normal((n, d)).astype(np.float32)
    path = str(tmp_path / "s.idx")
    libs.build_index_gpu(base, np.arange(n, dtype=np.int32), path, ef_c=32)
    return base, libs.Index.load(path)


@pytest.mark.parametrize("nq", [20, 2000])
def test_first_calls_beside_another_threads_capture(libs, tmp_path, nq):
    """The page-locked block, or the staging buffers of a larger call, are allocated while another thread captures a graph:
    the call works and the capture is not spoilt."""
    base, gix = _small(libs, tmp_path)
    side = torch.cuda.Stream()
    # the stream's scratch is there; pinned buffers need no block
    pinned = [torch.from_numpy(x).pin_memory() for x in (base[:nq] + 0.1, np.zeros(nq, np.int32), np.full(nq, 900, np.int32))]
    held = [torch.empty((nq, 5), dtype=t).pin_memory() for t in (torch.int32, torch.float32)]
    want = [x.clone() for x in gix.search_host(*pinned, 5, 32, out_ids=held[0], out_dists=held[1], stream=side)]
    plain = [x.clone() for x in pinned]
    out = [torch.zeros((nq, 5), dtype=t) for t in (torch.int32, torch.float32)]
    x, errors = torch.zeros(1000, device="cuda"), []
    torch.cuda.synchronize()

    def call():
        try:
            gix.search_host(*plain, 5, 32, out_ids=out[0], out_dists=out[1], stream=side)
        except libs.FrogError as e:
            errors.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x += 1
        t = threading.Thread(target=call)
        t.start()
        t.join()
        x += 1
    graph.replay()
    torch.cuda.synchronize()
    assert not errors and float(x[0]) == 2.0
    assert torch.equal(out[0], want[0]) and torch.equal(out[1], want[1])
    graph.reset()
    gix.close()
