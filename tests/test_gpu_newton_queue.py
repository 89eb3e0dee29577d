"""The mixed inversion's FP64 queue (csrc/pr_kernels.cuh): cells of the
pseudo-boiling band, all of which wait in a block's queue, at sizes around the
block (one cell, a block less and more one, several rounds), alone and among
cells that do not queue.  A queued cell's T is the FP64 inversion of the same
FP32 inputs rounded to FP32: within 2^-23 of the FP64 kernel's."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 257, 4099])
@pytest.mark.parametrize("share", [1.0, 0.3])
def test_band_cells_in_the_queue(prlib, cuda, n, share):
    import torch
    from paper_2312_04830_gb300 import binding
    ctx = binding.PropertyContext(W.species_table())
    rng = np.random.default_rng(n)
    T = np.where(rng.uniform(size=n) < share, rng.uniform(160.0, 175.0, n), rng.uniform(400.0, 900.0, n))
    Y = np.zeros((9, n))
    Y[1] = 1.0   # oxygen at 6 MPa: cp far above three times the ideal gas's around 163 K
    d = lambda a: torch.as_tensor(a, dtype=torch.float64, device=cuda)
    p = np.full(n, 6e6)
    o, st = ctx.props(d(T), d(p), d(Y))
    assert (st == 0).all()
    h32 = o[2].float()
    guess = d(np.clip(T * 1.02, 100.0, 3500.0)).float()
    Tm, sm, it = ctx.T_from_h(h32, d(p).float(), d(Y).float(), guess, "mixed")
    T64, s64, _ = ctx.T_from_h(h32.double(), d(p), d(Y), guess.double(), "fp64")
    torch.cuda.synchronize()
    assert (sm == 0).all() and (s64 == 0).all() and (it >= 1).all()
    band = o[3] > 3.2 * 918.0   # comfortably inside the band: cp over 3.2 times O2's ideal-gas cp at 165 K
    err = ((Tm.double() - T64) / T64).abs()
    assert float(err[band].max() if band.any() else 0.0) <= 2.0 ** -23
    assert float(err.max()) <= 2e-5
    ctx.close()
