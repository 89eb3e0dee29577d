"""The FP64 inversion next to critical points, where the cubic's three roots
meet and Newton's polish of the chosen one divides by a derivative that
vanishes: species alone in their cells, T and p within 0 to 1e-5 of their
critical values, among them critical temperatures that FP32 holds exactly (the
warm start then ends on them); against the FP64-only inversion.  h(T) rises
steeply there (cp -> infinity), so T is well determined: 1e-10, the parity bar
of the FP64 paths, and the same status."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exact", [False, True])
def test_near_critical(prlib, cuda, exact):
    import torch
    from paper_2312_04830_gb300 import binding
    sp = W.species_table()
    if exact:
        sp.Tc = np.round(sp.Tc * 4.0) / 4.0
    d0 = np.concatenate([[0.0], np.logspace(-12, -5, 29)])
    dT, dp = (v.ravel() for v in np.meshgrid(np.concatenate([d0, -d0]), np.concatenate([d0, -d0])))
    m = dT.size
    T = np.concatenate([sp.Tc[k] * (1.0 + dT) for k in range(9)])
    p = np.concatenate([sp.pc[k] * (1.0 + dp) for k in range(9)])
    Y = np.zeros((9, T.size))
    for k in range(9):
        Y[k, k * m:(k + 1) * m] = 1.0
    keep = T > 70.0   # the bracket's lower end is 60 K
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=cuda)
    T, p, Y = d(T[keep]), d(p[keep]), d(Y[:, keep])
    ctx, gen = binding.PropertyContext(sp), binding.PropertyContext(sp, newton_fp64_only=True)
    h = ctx.props(T, p, Y)[0][2].contiguous()
    for f in (1.0, 1.001, 1.05):
        guess = (T * f).contiguous()
        Tg, st, _ = ctx.T_from_h(h, p, Y, guess)
        Tn, sn, _ = gen.T_from_h(h, p, Y, guess)
        torch.cuda.synchronize()
        assert torch.equal(st, sn), (f, int((st != sn).sum()))
        ok = st == 0
        err = ((Tg - Tn) / Tn).abs()[ok]
        assert ok.double().mean() > 0.9 and float(err.max()) <= 1e-10, (f, float(err.max()), int((err > 1e-10).sum()))
    ctx.close()
    gen.close()
