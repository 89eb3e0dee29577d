"""A species table with one outsized constant: the inversion's fixed-point sums
carry a unit of their table's largest constant, so such a table keeps the
general form, and cells without that species keep their digits (the FP64-only
inversion within 1e-10, the parity bar of the FP64 paths)."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what", ["nasa_lo", "nasa_hi", "a6", "b", "a", "W"])
def test_outsized_constant(prlib, cuda, what):
    import torch
    from paper_2312_04830_gb300 import binding
    sp = W.species_table()
    for f in ("nasa_lo", "nasa_hi", "pc", "Tc", "W"):
        setattr(sp, f, getattr(sp, f).copy())
    big = 1e10
    if what in ("nasa_lo", "nasa_hi"):
        getattr(sp, what)[8, 4] *= big
    elif what == "a6":
        sp.nasa_lo[8, 5] *= big
    elif what == "b":
        sp.pc[8] /= big
    elif what == "a":
        sp.Tc[8] *= 1e20
        sp.pc[8] *= 1e20
    else:
        sp.W[8] /= big
    n = 5000
    T, p, Y = W.uniform_cells(n, seed=8)
    Y = Y.copy()
    Y[8] = 0.0
    Y /= Y.sum(axis=0)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    T, p, Y = d(np.clip(T, 400.0, 3400.0)), d(p), d(Y)
    ctx, gen = binding.PropertyContext(sp), binding.PropertyContext(sp, newton_fp64_only=True)
    h = ctx.props(T, p, Y)[0][2].contiguous()
    guess = (T * 1.03).clamp(100.0, 3500.0)
    Tg, st, _ = ctx.T_from_h(h, p, Y, guess)
    Tn, sn, _ = gen.T_from_h(h, p, Y, guess)
    torch.cuda.synchronize()
    assert torch.equal(st, sn) and (st == 0).double().mean() > 0.99
    away = (st == 0) & ((Tn - 1000.0).abs() > 1e-3)   # h(T) steps at the NASA-7 switch
    assert float(((Tg - Tn) / Tn)[away].abs().max()) <= 1e-10
    ctx.close()
    gen.close()
