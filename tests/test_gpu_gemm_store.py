"""Row pieces of the GEMM epilogue: BF16 results that start on 8 or 16 bytes, partial row and
column blocks, and nothing written beside them."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N", [(1, 16), (31, 32), (33, 48), (129, 272), (200, 240)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_results_at_any_alignment(M, N, mode):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_09900_gb300 import build
    build.build()
    import paper_2205_09900_gb300 as fp
    fp.load()
    K = 72
    g = torch.Generator().manual_seed(M + N)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16).cuda()
    Bt = torch.randn(N, K, generator=g).to(torch.bfloat16).cuda()
    bias = torch.randn(N, generator=g).cuda()
    z = torch.randn(M, N, generator=g).cuda()
    out = []
    for off in (8, 12):   # elements: 16 and 24 bytes into the buffers
        bufs = [torch.full((M * N + 32,), 7.0, device="cuda", dtype=t) for t in (torch.float32, torch.bfloat16)]
        C = [bufs[0][8:8 + M * N].view(M, N), bufs[1][off:off + M * N].view(M, N)]
        zc = z.clone()
        fp.gemm_bf16(A, Bt, bias, mode, zc, C[0], C[1])
        out.append([t.clone() for t in C] + [zc])
        for b, o in zip(bufs, (8, off)):
            assert torch.all(b[:o] == 7) and torch.all(b[o + M * N:] == 7)
    for p, q in zip(*out):
        assert torch.equal(p, q)   # the same arithmetic: the same bits
    assert torch.equal(out[0][0].to(torch.bfloat16), out[0][1])
