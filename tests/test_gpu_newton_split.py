"""The FP64 inversion's two-launch form (csrc/pr_inst_fix9.cu, more cells than
one wave of its single kernel) against the single kernel on the same cells:
both start the FP64 evaluation from FP32 iterations of the same cells, whose
results may differ by FP32 rounding, and accept within 1e-12 T of the root or
iterate to 1e-13, so T agrees to 1e-11; refused guesses, bad mass fractions,
temperatures out of the bracket, an in-place T_guess, and arrays that overlap
the result (which keep the single kernel)."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N = 152 * 8 * 128 + 77   # above one wave of any occupancy of the single kernel (at most eight blocks an SM)


def _inputs(cuda):
    import torch
    T, p, Y = W.uniform_cells(N, seed=77)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    return d(T), d(p), d(Y)


def test_two_launches_equal_one(prlib, cuda):
    import torch
    from paper_2312_04830_gb300 import binding
    ctx = binding.PropertyContext(W.species_table())
    T, p, Y = _inputs(cuda)
    h = ctx.props(T, p, Y)[0][2].contiguous()
    guess = (T * 1.04).clamp(100.0, 3500.0)
    guess[5], guess[6], guess[7] = float("nan"), float("inf"), 1e9
    h[8], h[9] = 1e12, float("nan")
    Y[0, 10] += 0.5
    Tg, st, it = ctx.T_from_h(h, p, Y, guess)
    one = [ctx.T_from_h(h[a:a + 30000].contiguous(), p[a:a + 30000].contiguous(), Y[:, a:a + 30000].contiguous(),
                        guess[a:a + 30000].contiguous()) for a in range(0, N, 30000)]
    T1, s1 = torch.cat([o[0] for o in one]), torch.cat([o[1] for o in one])
    assert torch.equal(st, s1)
    assert st[5] == 4 and st[6] == 4 and st[9] == 4 and st[10] == 4 and st[7] == 0 and st[8] == 2
    ok = st == 0
    assert float(ok.double().mean()) > 0.99
    assert float(((Tg - T1)[ok] / T1[ok]).abs().max()) <= 1e-11
    assert (it[ok] >= 1).all()
    # in place: the result over the guess
    g2 = guess.clone()
    Tb, sb, _ = ctx.T_from_h(h, p, Y, g2, T_out=g2)
    assert torch.equal(sb, st) and torch.equal(Tb[ok], Tg[ok])
    # the result over h*: the single kernel
    h2 = h.clone()
    Tc, sc, _ = ctx.T_from_h(h2, p, Y, guess, T_out=h2)
    assert torch.equal(sc, st)
    assert float(((Tc - Tg)[ok] / Tg[ok]).abs().max()) <= 1e-11
    ctx.close()
