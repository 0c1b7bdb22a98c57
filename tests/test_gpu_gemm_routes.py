"""Products of more than 128 rows around the lines between single CTAs and CTA
pairs: tiles around half a wave and one wave of 128 x 128, K around 512 and
2048 a slice, outputs that leave row by row and by TMA.  Each element within the
error of an FP32 sum of its K products in any order (K u / (1 - K u) times the
sum of their magnitudes, u = 2^-23, which also covers a truncating adder), plus
the rounding of the epilogue."""
import pytest
import torch

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("M,N,K,splits", [(1216, 1024, 504, 1), (1217, 1024, 504, 1), (2432, 1024, 520, 1),
                                          (2433, 1024, 520, 1), (2433, 1024, 448, 1), (2433, 1003, 448, 1),
                                          (2433, 1003, 520, 1), (300, 300, 2048, 1), (300, 300, 2120, 1),
                                          (300, 301, 4240, 2), (300, 301, 4096, 2), (2560, 1000, 4240, 2),
                                          (140, 20001, 72, 1)])
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


@pytest.mark.parametrize("M,N,K,epilogue,pairs", [
    (8192, 8192, 64, 1, False), (8192, 8192, 64, 0, True), (8192, 8192, 512, 1, True),  # BF16 rows, short and not
    (2048, 1003, 256, 0, False), (2048, 1004, 256, 0, True),                            # FP32 rows on 16 bytes or not
    (1000, 1003, 256, 1, True),                                                         # less than half a wave
    (2048, 128, 8192, 0, False), (2048, 128, 2048, 0, True), (8192, 4096, 4096, 0, True)])  # one wave of deep tiles
def test_kernel_of_a_product(M, N, K, epilogue, pairs):
    from torch.profiler import ProfilerActivity, profile

    from paper_1705_02403_gb300 import _native as N_
    A = torch.zeros(M, K, device="cuda", dtype=torch.bfloat16)
    B = torch.zeros(N, K, device="cuda", dtype=torch.bfloat16)
    N_.gmt_gemm_bf16(A, B, epilogue)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        N_.gmt_gemm_bf16(A, B, epilogue)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "gemm_" in e.name]
    if not names:
        pytest.skip("the profiler records no kernels here")
    assert len(names) == 1 and ("gemm_pair" in names[0]) == pairs
