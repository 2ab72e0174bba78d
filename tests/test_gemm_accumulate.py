"""Accumulating products keep subnormal values (GPU), on one SM (M <= 128) and on
pairs (M > 128): C += A B with A = 0 leaves every subnormal entry of C as it was, and
1.5 2^-126 plus a product of -2^-126 is 2^-127."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [100, 257])
def test_accumulate_keeps_subnormals(M):
    import torch
    import paper_2604_08542_gb300 as ttt
    N, K = 4096, 64
    g = torch.Generator(device="cuda").manual_seed(M)
    layer = ttt.TTT(1, 256, 256, dtype=torch.bfloat16)
    st = torch.cuda.current_stream().cuda_stream

    def accumulate(a, b, c):
        assert ttt.scal3r_ttt_gemm(layer.handle, a.data_ptr(), K, 1, b.data_ptr(), K, 1, c.data_ptr(), N, 1, 1, M, N,
                                   K, None, 0, st) == 0
        return c.view(torch.int32)

    a = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    b = torch.randn((N, K), generator=g, device="cuda").to(torch.bfloat16)
    bits = torch.randint(1, 1 << 23, (M, N), generator=g, device="cuda", dtype=torch.int32)   # subnormals
    assert torch.equal(accumulate(a, b, bits.clone().view(torch.float32)), bits)
    a[:, 0], b[:] = -(2.0 ** -63), 0
    b[:, 0] = 2.0 ** -63
    c = accumulate(a, b, torch.full((M, N), 1.5 * 2.0 ** -126, device="cuda"))
    assert (c == 1 << 22).all()   # 2^-127
    assert layer.status() == 0
