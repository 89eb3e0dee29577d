"""The GEMMs of two and more M-tiles run on CTA pairs, those of one on single
CTAs: both give the same bits, odd M-tile counts and ragged rows included."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(prlib, cuda, species):
    from paper_2312_04830_gb300 import binding
    c = binding.PropertyContext(species)
    yield c
    c.close()


@pytest.mark.parametrize("M,N,K", [(129, 128, 64), (256, 256, 64), (384, 384, 320), (641, 512, 128),
                                   (20000, 1024, 64)])
def test_pair_equals_single(prlib, cuda, M, N, K):
    import torch
    from paper_2312_04830_gb300 import binding
    g = torch.Generator(device="cpu").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16).to(cuda)
    B = torch.randn(N, K, generator=g).to(torch.bfloat16).to(cuda)
    D, err = binding.gemm_bf16(A, B)
    for r in (0, 128, (M - 1) // 256 * 256, (M - 1) // 128 * 128):
        one, e1 = binding.gemm_bf16(A[r:r + 128].contiguous(), B)
        assert torch.equal(D[r:r + 128], one), r
        assert int(e1.item()) == 0
    assert int(err.item()) == 0


@pytest.mark.parametrize("width", [128, 256, 512, 1024])
def test_pairs_in_training_and_layerwise_inference(ctx, cuda, width):
    """A batch's gradient is the mean of its 128-row parts' gradients.  512
    rows: the loss scale is a power of two apart, so dz has the same digits and
    only the FP32 sums' order differs (512 terms: 512 x 2^-24 of the sums of
    absolute values, 1e-3 of the result at a cancellation of 30).  384 rows (an
    odd M-tile count, stale rows above it in the buffers): dz is rounded to
    BF16 at another scale in every layer, 2^-9 each: 2e-2."""
    import torch
    from paper_2312_04830_gb300 import binding
    g = torch.Generator(device="cpu").manual_seed(width)
    x = torch.rand(11, 512, generator=g) + 0.1
    x[0] = 300.0 + 2000.0 * x[0]
    x[1] = 1e7 * x[1]
    x[2:] /= x[2:].sum(0)
    y = torch.randn(6, 512, generator=g)
    x, y = x.to(cuda), y.to(cuda)
    sg = binding.Surrogate(ctx, width=width, hidden_layers=3, max_batch=512, infer_chunk=512, seed=3)
    sg.fit_normalization(x, y)

    def grad(lo, hi):
        return sg.loss_grad(x[:, lo:hi].contiguous(), y[:, lo:hi].contiguous(), hi - lo)[1].double()
    parts = [grad(i, i + 128) for i in range(0, 512, 128)]
    for n, tol in ((512, 1e-3), (384, 2e-2)):
        mean = sum(parts[:n // 128]) / (n // 128)
        assert float((grad(0, n) - mean).norm() / mean.norm()) < tol, n
    sg.set_fused_infer(False)
    for n in (130, 300, 512):
        out, _ = sg.infer(x[0, :n].contiguous(), x[1, :n].contiguous(), x[2:, :n].contiguous())
        for r in range(0, n, 128):
            s = slice(r, min(r + 128, n))
            one, _ = sg.infer(x[0, s].contiguous(), x[1, s].contiguous(), x[2:, s].contiguous())
            assert np.array_equal(out[:, s].cpu().numpy(), one.cpu().numpy(), equal_nan=True), (n, r)
    sg.sync_status()
    sg.close()


def test_captured_steps(ctx, cuda):
    """Training steps under stream capture: two steps in a graph (learning rate
    zero, so every step has the same loss) give the loss of one outside it."""
    import torch
    from paper_2312_04830_gb300 import binding
    g = torch.Generator(device="cpu").manual_seed(9)
    x = torch.rand(11, 1024, generator=g) + 0.1
    x[0], x[1] = 300.0 + 2000.0 * x[0], 1e7 * x[1]
    x[2:] /= x[2:].sum(0)
    x, y = x.to(cuda), torch.randn(6, 1024, generator=g).to(cuda)
    sg = binding.Surrogate(ctx, width=256, hidden_layers=2, max_batch=1024, infer_chunk=1024, seed=3)
    sg.fit_normalization(x, y)
    loss = torch.zeros(2, device=cuda)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        sg.train_step(x, y, 1024, 0.0, sample_seed=5, loss_out=loss, stream=st)
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            for _ in range(2):
                sg.train_step(x, y, 1024, 0.0, sample_seed=5, loss_out=loss[1:], stream=st)
        for _ in range(3):
            graph.replay()
    torch.cuda.synchronize()
    assert float(loss[0]) == float(loss[1]) > 0.0
    sg.sync_status()
    sg.close()
