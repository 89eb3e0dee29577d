"""Blocks of one and two warps for calls that fill at most one such block an SM:
every cell has the bits it has in a call of whole blocks."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "mixed"])
def test_small_calls_equal_large(prlib, cuda, prec):
    import torch
    from paper_2312_04830_gb300 import binding
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 64 * sms + 129
    T, p, Y = W.training_states(n, seed=5)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=cuda).to(torch.float64 if prec == "fp64" else torch.float32)
    T, p, Y = d(T), d(p), d(Y)
    ctx = binding.PropertyContext(W.species_table())

    def calls(m):
        Tm, pm, Ym = T[:m].contiguous(), p[:m].contiguous(), Y[:, :m].contiguous()
        o, st = ctx.props(Tm, pm, Ym, prec)
        Th = ctx.T_from_h(o[2].contiguous(), pm, Ym, (0.97 * Tm).contiguous(), prec)
        return [*o, st, *Th]
    big = calls(n)
    for m in (1, 31, 33, 1000, 32 * sms, 32 * sms + 1, 64 * sms, 64 * sms + 1):
        for a, b in zip(calls(m), big):
            assert np.array_equal(a.cpu().numpy(), b[:m].cpu().numpy(), equal_nan=True), m
    ctx.close()
