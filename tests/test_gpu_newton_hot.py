"""Roots above the fixed-point range (4096 K) take the FP64 inversion's one-step
acceptance too, from one general evaluation: almost every cell in one FP64
evaluation, in the single kernel and in the two launches, T as the FP64-only
inversion's to 1e-11 (both within 1e-12 of the root or iterated to 1e-13), next
to cells below the range's end."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [500, 152 * 8 * 128 + 77])   # one launch; two
def test_one_evaluation_above_4096(prlib, cuda, n):
    import torch
    from paper_2312_04830_gb300 import binding
    rng = np.random.default_rng(n)
    T = np.where(np.arange(n) % 3 == 0, rng.uniform(3900.0, 4300.0, n), rng.uniform(4100.0, 4900.0, n))
    T[:4] = [4096.0, np.nextafter(4096.0, 0.0), 4096.0 * (1 + 1e-7), 4096.0 * (1 - 1e-7)]
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    T, p, Y = d(T), d(np.where(np.arange(n) % 2 == 0, 1e5, 1e7)), d(W.dirichlet_half(rng, 9, n))
    ctx = binding.PropertyContext(W.species_table())
    gen = binding.PropertyContext(W.species_table(), newton_fp64_only=True)
    h = ctx.props(T, p, Y)[0][2].contiguous()
    guess = (T * 1.01).contiguous()
    Tg, st, it = ctx.T_from_h(h, p, Y, guess)
    Tn, sn, _ = gen.T_from_h(h, p, Y, guess)
    torch.cuda.synchronize()
    assert (st == 0).all() and torch.equal(st, sn)
    assert float(((Tg - Tn) / Tn).abs().max()) <= 1e-11
    assert float((it == 1).double().mean()) > 0.98
    ctx.close()
    gen.close()
