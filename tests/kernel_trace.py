"""Which kernels a call launches, by name (with template arguments), for tests
that have to know which of several forms ran."""
import time

import pytest


def traced(call):
    """Names of the CUDA calls, kernels and copies of call()."""
    import torch
    from torch.profiler import ProfilerActivity, profile

    for _ in range(3):  # the first trace of a process can come back empty
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            time.sleep(0.02)  # kernels at the very ends of a trace are dropped
            call()
            torch.cuda.synchronize()
            time.sleep(0.02)
        names = [e.name for e in p.events()]
        if any("stag::" in n for n in names):
            return names
    pytest.skip("no kernel trace on this machine")


def launched(call):
    """Names of the library's kernels that call() launches."""
    return [n.split("(")[0].replace("stag::", "") for n in traced(call) if n.startswith(("void stag::", "stag::"))]
