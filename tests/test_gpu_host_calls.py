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
