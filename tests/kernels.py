"""Which kernels of the library a call launches, for tests that are about one of several forms."""
import re

import torch


def launched(call):
    """(result of call(), the names k_... of the kernels that ran, without template arguments)."""
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA], acc_events=True) as trace:
        result = call()
        torch.cuda.synchronize()
    found = (re.search(r"psattn::(k_\w+)", e.name) for e in trace.events())
    return result, {m.group(1) for m in found if m}
