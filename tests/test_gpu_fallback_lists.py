"""The surrogate's FP64 fallback on lists of all lengths around its warps, its
blocks and its grid: every listed cell is written (the output starts as NaN),
with the FP64 properties of the same FP32 inputs (one rounding to FP32, and the
integer-pipe forms compiled into another kernel: 2^-22)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 608, 19456 + 33, 77824 - 1, 77824 + 5, 200003])
def test_every_listed_cell(prlib, cuda, species, n):
    import torch
    from paper_2312_04830_gb300 import binding, workloads as W
    ctx = binding.PropertyContext(species)
    T, p, Y = W.training_states(4096, seed=2)
    d = lambda a: torch.as_tensor(a, device=cuda).float().contiguous()
    x = torch.cat([d(T)[None], d(p)[None], d(Y)])
    y = ctx.props(x[0].contiguous(), x[1].contiguous(), x[2:].contiguous(), "fp32")[0]
    sg = binding.Surrogate(ctx, width=128, hidden_layers=1, max_batch=128, infer_chunk=1 << 18, seed=1)
    sg.fit_normalization(x, y)
    g = torch.Generator(device="cpu").manual_seed(n)
    Tn = (400.0 + 2500.0 * torch.rand(n, generator=g)).to(cuda)
    pn = torch.full((n,), 3e7, device=cuda)   # outside the hull
    z = torch.randn(9, n, generator=g) ** 2
    Yn = (z / z.sum(0)).to(cuda).contiguous()
    out = torch.full((6, n), float("nan"), device=cuda)
    _, fb = sg.infer(Tn, pn, Yn, out=out)
    sg.sync_status()
    ref, st = ctx.props(Tn.double(), pn.double(), Yn.double())
    assert (fb == 1).all()
    ok = st == 0
    assert ok.double().mean() > 0.9
    scale = ref.abs()
    scale[2] = torch.maximum(scale[2], ref[3].abs() * Tn.double())
    assert float(((out.double() - ref).abs() / scale)[:, ok].max()) <= 2.0 ** -22
    sg.close()
    ctx.close()
