"""Which kernels calls launch, by torch's profiler, in a process of its own: `record_launches.py index queries.npz steps` prints
for every step the (name, threads of a CTA) of this library's kernels.  A session of the profiler some seconds after another
one of the same process may record no kernels at all; hence the process, and the pauses, as what seems to lie outside a
session's window is dropped."""
import json
import os
import sys
import tempfile
import time
import warnings

import numpy as np
import torch
from torch.profiler import ProfilerActivity, profile

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import paper_2608_16491_b200 as libs                                    # noqa: E402


def main(index, queries, steps):
    gix = libs.Index.load(index)
    gix.enable_f16()
    data = np.load(queries)
    q, lo, hi = (torch.from_numpy(data[x]).cuda() for x in ("q", "lo", "hi"))
    other = torch.cuda.Stream()
    kept = [torch.empty((len(q), 10), dtype=t, device="cuda") for t in (torch.int32, torch.float32)]
    trace = os.path.join(tempfile.mkdtemp(), "trace.json")
    for step in steps:
        part = [x[:step["nq"]] for x in (q, lo, hi)]

        def call():
            if step.get("beside"):                                       # some milliseconds of the general kernel
                gix.search(q, lo, hi, 10, 512, stream=other, out_ids=kept[0], out_dists=kept[1],
                           params=libs.Params(budget=64, visited=libs.VISITED_HASH))
            if "ef" in step:
                return gix.search(*part, 10, step["ef"], params=libs.Params(budget=step["budget"], storage=step.get("storage", 0)))
            return gix.exact_search(*part, step["k"])

        for _ in range(3):                                               # scratch is there, kernels are loaded
            call()
            torch.cuda.synchronize()
        with warnings.catch_warnings():
            warnings.simplefilter("ignore")
            with profile(activities=[ProfilerActivity.CUDA]) as prof:
                time.sleep(0.02)
                call()
                torch.cuda.synchronize()
                time.sleep(0.02)
        prof.export_chrome_trace(trace)
        with open(trace) as f:
            events = json.load(f)["traceEvents"]
        found = [(e["name"], e["args"]["block"][0]) for e in events
                 if e.get("cat") == "kernel" and ("frog_" in e["name"] or "filter_" in e["name"])]
        print("LAUNCHES", json.dumps(found))


if __name__ == "__main__":
    main(sys.argv[1], sys.argv[2], json.loads(sys.argv[3]))
