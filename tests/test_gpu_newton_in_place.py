"""The inversion with its result over one of its own inputs: every cell's
inputs are read before its result is written, so T, status and iteration count
have the bits of the call into an array of its own.  Cells of the
pseudo-boiling band (queued and solved again), cells that fail, refused cells
and, in mixed precision, queued cells whose mass fractions pass the sum check
in FP32 and not in FP64 (the FP32 result stands)."""
import numpy as np
import pytest

from paper_2312_04830_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp32", "fp64"])
@pytest.mark.parametrize("n", [129, 4099])
@pytest.mark.parametrize("over", ["h", "p", "guess", "Y"])
def test_result_over_an_input(prlib, cuda, prec, n, over):
    import torch
    from paper_2312_04830_gb300 import binding
    ctx = binding.PropertyContext(W.species_table())
    rng = np.random.default_rng(n)
    T = np.where(rng.uniform(size=n) < 0.4, rng.uniform(160.0, 175.0, n), rng.uniform(400.0, 900.0, n))
    Y = np.zeros((9, n))
    Y[1] = 1.0   # oxygen at 6 MPa: the band is around 163 K
    d = lambda a: torch.as_tensor(a, dtype=torch.float64, device=cuda)
    p = np.full(n, 6e6)
    h = ctx.props(d(T), d(p), d(Y))[0][2].cpu().numpy()
    h[3], h[4], h[5] = 1e12, np.nan, -1e12
    Y[0, 6] = 0.5
    guess = np.clip(T * 1.02, 100.0, 3500.0)
    guess[7] = np.inf
    # FP32 sum 1 + 8 ulp (9.54e-7), exact sum 1 + 1.003e-6
    Y[1, 8:12], Y[0, 8:12], h[8:12] = 1.0 + 8 * 2.0 ** -23, 5e-8, h[8:12] * (1.0 + 8 * 2.0 ** -23)
    dt = torch.float64 if prec == "fp64" else torch.float32
    a = {"h": d(h).to(dt), "p": d(p).to(dt), "Y": d(Y).to(dt), "guess": d(guess).to(dt)}
    call = lambda b, out: ctx.T_from_h(b["h"], b["p"], b["Y"], b["guess"], prec, T_out=out)
    T1, s1, i1 = call(a, None)
    b = {k: v.clone() for k, v in a.items()}
    T2, s2, i2 = call(b, b["Y"][1] if over == "Y" else b[over])
    torch.cuda.synchronize()
    bits = torch.int64 if prec == "fp64" else torch.int32
    assert torch.equal(s1, s2) and torch.equal(i1, i2)
    assert torch.equal(T1.view(bits), T2.view(bits))
    assert (s1[12:] == 0).all() and s1[4] == 4 and s1[6] == 4 and s1[7] == 4
    ctx.close()
