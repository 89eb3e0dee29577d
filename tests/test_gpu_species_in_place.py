"""The per-species outputs over the mass fractions: every cell's Y is read
before either output of the cell is written, so both outputs have the bits of
the call into arrays of their own; inside and outside the fixed-point range,
refused cells, species alone in their cells."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("over", ["hk", "Dk"])
@pytest.mark.parametrize("both", [True, False])
def test_output_over_the_mass_fractions(prlib, cuda, prec, over, both):
    import torch
    from paper_2312_04830_gb300 import binding
    ctx = binding.PropertyContext(W.species_table())
    n = 517
    T, p, Y = W.uniform_cells(n, seed=3)
    T, Y = T.copy(), Y.copy()
    T[1], T[2], T[3] = 20.0, 9000.0, -1.0
    Y[:, 4], Y[2, 4] = 0.0, 1.0
    Y[0, 5] += 0.5
    dt = torch.float64 if prec == "fp64" else torch.float32
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=cuda).to(dt)
    T, p, Y = d(T), d(p), d(Y)
    want = {"hk": True, "Dk": True} if both else {"hk": over == "hk", "Dk": over == "Dk"}
    hk, Dk, st = ctx.species_props(T, p, Y, prec, **want)
    Y2 = Y.clone()
    h2, D2, s2 = ctx.species_props(T, p, Y2, prec, **{**want, over: Y2})
    torch.cuda.synchronize()
    bits = torch.int64 if prec == "fp64" else torch.int32
    assert torch.equal(st, s2) and st[3] == 4 and st[5] == 4
    for a, b in ((hk, h2), (Dk, D2)):
        assert a is None or torch.equal(a.view(bits), b.view(bits))
    ctx.close()
