"""The kernels that a call launches, by name (for tests of which form a call
takes, where the forms give the same bits)."""
import torch

_warm = False


def _profiled(fn):
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        out = fn()
        torch.cuda.synchronize()
    return out, [ev.key for ev in prof.key_averages()]


def kernel_names(fn):
    """fn() and the names of its kernels (a process's first trace may miss some)."""
    global _warm
    for _ in range(0 if _warm else 3):
        _, names = _profiled(lambda: torch.zeros(8, device="cuda").add_(1))
        _warm = _warm or any("elementwise" in n for n in names)
    return _profiled(fn)
