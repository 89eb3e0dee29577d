"""The FP64 inversion's first evaluation in fixed point (csrc/pr_fix9.cuh) on
species alone in their cells with a mass fraction within rounding of 1, where
the mole fraction reaches the end of its 62 bits: Y = 1 + j ulp for each
species, in the single kernel and in the two launches, against the FP64-only
inversion.  Both accept within 1e-12 T of the root or iterate to 1e-13: 1e-11,
as for the two forms of the kernel."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_side", [3000, 6000])   # 54 009 cells: one launch; 108 009: two
def test_species_alone_near_one(prlib, cuda, per_side):
    import torch
    from paper_2312_04830_gb300 import binding
    sp = W.species_table()
    j = np.arange(-per_side, per_side + 1)
    y = 1.0 + np.where(j < 0, j * 2.0 ** -53, j * 2.0 ** -52)
    n = 9 * j.size
    Y = np.zeros((9, n))
    for k in range(9):
        Y[k, k * j.size:(k + 1) * j.size] = y
    rng = np.random.default_rng(per_side)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    T, p, Y = d(rng.uniform(1100.0, 3000.0, n)), d(np.where(np.arange(n) % 2 == 0, 1e5, 1e7)), d(Y)
    ctx, gen = binding.PropertyContext(sp), binding.PropertyContext(sp, newton_fp64_only=True)
    h = ctx.props(T, p, Y)[0][2].contiguous()
    guess = (T * 1.03).clamp(100.0, 3500.0)
    Tg, st, it = ctx.T_from_h(h, p, Y, guess)
    Tn, sn, _ = gen.T_from_h(h, p, Y, guess)
    torch.cuda.synchronize()
    assert torch.equal(st, sn) and (st == 0).all()
    assert float(((Tg - Tn) / Tn).abs().max()) <= 1e-11
    ctx.close()
    gen.close()
