"""GEMMs on CTA pairs (two or more M-tiles and K of 2048 and more) against
single CTAs (128 rows at a time), bit for bit: pairs that take several tiles,
so that the double-buffered accumulator and the stage ring come round, odd
M-tile counts and ragged rows, every row compared; and smaller K, on single
CTAs that take several tiles."""
import pytest

pytestmark = pytest.mark.gpu


# tiles of 128 or 256 columns; (20000, 1024, 320): 79 pair rows x 4 tiles on 76 pairs;
# (40000, 128, 192): 157 pair rows, the last one's second M-tile missing (313 M-tiles)
@pytest.mark.parametrize("M,N,K", [(129, 128, 128), (256, 256, 192), (20000, 1024, 320), (40000, 128, 192),
                                   (19999, 512, 1024), (20000, 1024, 64), (129, 128, 2048), (256, 256, 2112),
                                   (20000, 1024, 2112), (40000, 128, 2048), (19999, 512, 4096)])
def test_every_row(prlib, cuda, M, N, K):
    import torch
    from paper_2312_04830_gb300 import binding
    g = torch.Generator(device="cpu").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16).to(cuda)
    B = torch.randn(N, K, generator=g).to(torch.bfloat16).to(cuda)
    D, err = binding.gemm_bf16(A, B)
    bad = torch.zeros(1, dtype=torch.int64, device=cuda)
    for r in range(0, M, 128):
        one, e1 = binding.gemm_bf16(A[r:r + 128].contiguous(), B)
        bad += (D[r:r + 128] != one).sum() + e1.sum()
    assert int(bad.item()) == 0 and int(err.item()) == 0
