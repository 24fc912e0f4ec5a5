"""A bounded wait of the BF16 GEMM that runs out at any point of its pipeline: the
launch drains what it issued, the call reports FP_ERR_TIMEOUT (or is done in time
and correct), and the next call with the default limit is correct.

The roles of the kernel wait for different things (the loader and the MMA issuer for
one stage of the K loop, the epilogue for a whole tile), so one may give up after
another has issued all its work: with at most four stages the loader waits for
nothing, and with a limit between a stage's and a tile's time only the epilogue's
wait runs out."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(512, 256, 64), (512, 256, 256), (300, 48, 4096), (512, 512, 4096),
                                   (45000, 256, 1024)])
def test_wait_runs_out_anywhere(fp, M, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randint(-2, 3, (M, K), generator=g, device="cuda").to(torch.bfloat16)
    Bt = torch.randint(-2, 3, (N, K), generator=g, device="cuda").to(torch.bfloat16)
    C = torch.empty(M, N, dtype=torch.float32, device="cuda")
    ref = (A.float() @ Bt.float().T)      # small integers: exact in FP32 whatever the order
    try:
        for ns in (1, 300, 1000, 2000, 4000, 8000, 16000, 50000):
            fp.set_wait_limit_ns(ns)
            for _ in range(5):
                C.fill_(float("nan"))
                try:
                    fp.gemm_bf16(A, Bt, C=C)
                except fp.FpError as e:
                    assert e.status == -4
                else:
                    assert torch.equal(C, ref)
    finally:
        fp.set_wait_limit_ns(0)
    fp.gemm_bf16(A, Bt, C=C)
    assert torch.equal(C, ref)
