"""The CTA-pair GEMM at the edges of its tiles: rows around 128 and 256, columns
around the tile widths, K of one block, a remainder and several slices.  Each
element must lie within the error of an FP32 sum of its K products in any order
(K u / (1 - K u) times the sum of their magnitudes, u = 2^-23, which also
covers a truncating adder), plus the rounding of the epilogue."""
import pytest
import torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("M", [129, 255, 256, 257, 513])
@pytest.mark.parametrize("N,K,splits", [(1, 8, 1), (31, 64, 1), (33, 72, 1), (224, 136, 1), (225, 520, 3), (256, 64, 1),
                                        (257, 1000, 1), (5000, 128, 2), (20000, 64, 1)])
def test_products_within_the_sum_bound(M, N, K, splits):
    from paper_1705_02403_gb300 import _native as N_
    g = torch.Generator(device="cuda").manual_seed(M * 31 + N * 7 + K)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16)
    bias = torch.randn(N, device="cuda", generator=g)
    exact = A.double() @ B.double().T
    u = 2.0 ** -23
    bound = K * u / (1 - K * u) * (A.double().abs() @ B.double().abs().T)
    for epilogue in (0, 1, 2):
        C, err = N_.gmt_gemm_bf16(A, B, epilogue, bias=bias if epilogue else None, splits=splits)
        assert int(err.item()) == 0
        want = exact if epilogue == 0 else exact + bias.double()
        tol = bound + 2.0 ** -24 * (want.abs() + bound)
        if epilogue == 1:  # ReLU moves values no further apart; BF16 keeps eight bits
            want, tol = want.relu(), tol + 2.0 ** -8 * (want.relu() + bound)
        assert bool(((C.double() - want).abs() <= tol).all())
