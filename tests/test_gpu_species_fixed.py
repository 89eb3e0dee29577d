"""The fixed-point form of the FP64 per-species outputs (csrc/pr_species.cu,
species_fix_kernel) at the edges of its range, against the FP64 oracle: the
temperatures 32 and 8192 K where it hands over to the general form, one to
nine species, species alone in their cells, and a table with an eps_kj below
its range (helium-like), which takes the general form.  Tolerance 1e-12: both
sides round some 60 times (1e-14), the oracle's powers and sums within 1e-14."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu
RTOL = 1e-12


def _check(ctx, orc, species, T, p, Y, cuda):
    import torch
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    hk, Dk, st = ctx.species_props(d(T), d(p), d(Y))
    torch.cuda.synchronize()
    ohk, oDk, ost = orc.species_props(species, T, p, Y)
    assert np.array_equal(st.cpu().numpy(), ost)
    ehk = np.abs(hk.cpu().numpy() - ohk) / np.maximum(np.abs(ohk), 1.0)
    eDk = np.abs(Dk.cpu().numpy() - oDk) / np.abs(oDk)
    assert ehk.max() <= RTOL and eDk.max() <= RTOL, (ehk.max(), eDk.max())


@pytest.mark.parametrize("n_species", [1, 2, 5, 9])
def test_range_edges(prlib, orc, cuda, n_species):
    from paper_2312_04830_gb300 import binding
    sp = W.species_table().subset(W.SPECIES[:n_species])
    ctx = binding.PropertyContext(sp)
    up, dn = np.nextafter(8192.0, 1e9), np.nextafter(32.0, 0.0)
    T = np.array([32.0, dn, 33.0, 8192.0, np.nextafter(8192.0, 0.0), up, 63.999999999999, 64.0, 999.9999999999999,
                  1000.0, 1e-3, 2e4, 120.0, 3500.0])
    T = np.concatenate([T, np.random.default_rng(3).uniform(30.0, 8300.0, 243)])   # 257 cells: two blocks and one more
    p = np.where(np.arange(T.size) % 2 == 0, 1e7, 1e5)
    Y = W.dirichlet_half(np.random.default_rng(4), n_species, T.size)
    Y[:, 5] = 0.0
    Y[n_species - 1, 5] = 1.0   # alone in its cell, outside the range
    Y[:, 20] = 0.0
    Y[0, 20] = 1.0              # and inside
    Y = np.ascontiguousarray(Y / Y.sum(axis=0))
    _check(ctx, orc, sp, T, p, Y, cuda)
    ctx.close()


def test_small_eps_takes_the_general_form(prlib, orc, cuda):
    from paper_2312_04830_gb300 import binding
    sp = W.species_table()
    sp.Tc = sp.Tc.copy()
    sp.Tc[5] = 5.2
    ctx = binding.PropertyContext(sp)
    T, p, Y = W.uniform_cells(300, seed=5)
    _check(ctx, orc, sp, T, p, Y, cuda)
    ctx.close()
