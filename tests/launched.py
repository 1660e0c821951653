"""Which of the library's kernels a call launches: tests that are about one form of a kernel make sure that it is the one that ran."""
import collections
import json
import os
import re
import tempfile

import torch
from torch.profiler import ProfilerActivity, profile

Launch = collections.namedtuple("Launch", "kernel blocks shared")  # name with template arguments; blocks; bytes of shared memory of each


def launched(call):
    """The kernels of this library that call() launches, in their order."""
    call()  # (loading of the kernels, first use of the device)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA, ProfilerActivity.CPU]) as p:
        call()
        torch.cuda.synchronize()
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "trace.json")
        p.export_chrome_trace(path)
        with open(path) as f:
            events = [e for e in json.load(f)["traceEvents"] if e.get("cat") == "kernel"]
    out = []
    for e in sorted(events, key=lambda e: e["ts"]):
        m = re.search(r"(cowa_\w+)(<[^>]*>)?", e["name"])
        if m:
            x, y, z = e["args"]["grid"]
            out.append(Launch(m.group(1) + (m.group(2) or "").replace(" ", ""), x * y * z, e["args"]["shared memory"]))
    assert out, "the profiler saw no kernel of the library"
    return out
