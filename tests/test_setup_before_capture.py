"""StepGraph's eager steps before a capture reach the kernels of large steps,
not only those of the few cells that it steps."""
import types

import pytest
import torch

from paper_2202_10647_gb300 import ionize, multistep


@pytest.mark.parametrize("window", [None, {"w_min": 2, "w_max": 6, "eps_grow": 1e-6}])
@pytest.mark.parametrize("flags", [ionize.ION_F32, ionize.ION_CONSERVATION_CHECK,
                                   ionize.ION_F64_PLAIN])
def test_priming_reaches_the_large_steps_kernels(flags, window, monkeypatch):
    """An FP32 step without a shape runs one cell per lane up to 400,000
    cells, an FP64 step up to 32 warps per SM; the default shape is (2, 8, 0)."""
    seen, sms = [], 152

    def step(sp, E, N, lo, hi, dt, dne, flags=0, window=None, **kw):
        seen.append((E.numel(), N.shape[1], None, flags, window))

    def step_batched(jobs, dt, flags=0, shape=None, window=None, **kw):
        (sp, E, N, *_), = jobs
        seen.append((E.numel(), N.shape[1], shape, flags, window))

    monkeypatch.setattr(ionize, "step", step)
    monkeypatch.setattr(ionize, "step_batched", step_batched)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    monkeypatch.setattr(torch.cuda, "get_device_properties",
                        lambda d: types.SimpleNamespace(multi_processor_count=sms))
    sp = types.SimpleNamespace(Z=7)
    multistep._prime(sp, flags, window, "cpu")
    assert all(f == flags and w == window for *_, f, w in seen)
    if flags & ionize.ION_F64_PLAIN:
        assert any(n > 32 * 32 * sms for n, *_ in seen)
    else:  # even rows: the single-species kernel; odd ones: the general one
        big = {ld % 2 for n, ld, shape, *_ in seen if shape == (2, 8, 0) or n > 400_000}
        assert big == {0, 1}
