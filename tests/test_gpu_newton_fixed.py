"""The FP64 inversion's first evaluation in fixed point (csrc/pr_fix9.cuh):
one to nine species, roots on both sides of the fixed-point range's end
(4096 K), of the NASA-7 switch and of the zeros of the species' alpha factors,
species alone in their cells, mass fractions at the limit of the sum check;
against the FP64 oracle's inversion within 1e-10 (the parity bar of the FP64
paths), the status equal.  Where the mass fractions do not sum to 1, h scales
with their sum in the library (sum Y/W times the molar value) and in the
oracle's ideal-gas part only, so those cells are compared with the library's
general form (the FP64-only inversion)."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_species", [1, 2, 5, 9])
def test_range_edges(prlib, orc, cuda, n_species):
    import torch
    from paper_2312_04830_gb300 import binding
    sp = W.species_table().subset(W.SPECIES[:n_species])
    rng = np.random.default_rng(n_species)
    kap = 0.37464 + 1.54226 * sp.omega - 0.26992 * sp.omega ** 2
    zeros = sp.Tc * ((1.0 + kap) / kap) ** 2   # alpha factor 0 of each species
    T = np.concatenate([[61.0, 999.0, 1001.0, 4095.9, 4096.0, 4097.0, 4990.0], zeros[zeros < 4900.0] * 1.0001,
                        rng.uniform(100.0, 4900.0, 250)])
    n = T.size
    p = np.where(np.arange(n) % 3 == 0, 1e5, 1e7)
    Y = W.dirichlet_half(rng, n_species, n)
    Y[:, 3] = 0.0
    Y[n_species - 1, 3] = 1.0
    Y[:, -1] = 1e-320          # subnormal traces
    Y[0, -1] = 1.0
    Y = np.ascontiguousarray(Y / Y.sum(axis=0))
    Y[:, -2] *= 1.0 + 0.9e-6   # inside the limit of 1e-6
    Y[:, -3] *= 1.0 + 1.1e-6   # and outside
    Y[0, -4] = -0.0
    Y[n_species - 1, -4] += 1.0 - Y[:, -4].sum()
    o, st = orc.props(sp, T, p, Y)
    h = o[2].copy()
    h[np.isnan(h)] = 0.0
    guess = np.clip(T * 1.05, 100.0, 3500.0)
    To, so, _ = orc.T_from_h(sp, h, p, Y, guess)
    ctx = binding.PropertyContext(sp)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    Tg, sg, it = ctx.T_from_h(d(h), d(p), d(Y), d(guess))
    torch.cuda.synchronize()
    Tg, sg = Tg.cpu().numpy(), sg.cpu().numpy()
    assert np.array_equal(sg, so)
    ok = so == 0
    assert ok.sum() > 0.9 * n and so[-3] == 4
    # a root inside the jump of h(T) at the NASA-7 switch is either side's
    gen = binding.PropertyContext(sp, newton_fp64_only=True)
    Tn, sn, _ = gen.T_from_h(d(h), d(p), d(Y), d(guess))
    assert np.array_equal(sn.cpu().numpy(), so)
    off = np.abs(Y.sum(axis=0) - 1.0) > 1e-12
    To = np.where(off, Tn.cpu().numpy(), To)
    gen.close()
    away = ok & (np.abs(To - 1000.0) > 1e-5)
    assert np.max(np.abs(Tg[away] - To[away]) / To[away]) <= 1e-10
    ctx.close()
