"""The wide path's product when every CTA pair takes several output tiles and the
last row block leaves warps without rows (GPU): 65 row blocks of 256 by 16 column
blocks for 76 pairs, the last block with 16 or 128 of its rows.  K is one or two
steps, so the launch is bound by its stores and a tile's staging buffers are
still being read when the next tile's accumulator is ready.

The operands are whole numbers up to 4 and K <= 128: every sum is below 2^24, so
float32 holds it exactly in any order and the outputs are compared to the bit
(the bfloat16 one is the rounded sum)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K", [(16400, 64), (16400, 128), (16512, 64)])
def test_rounds_of_tiles_with_a_clipped_last_block(M, K):
    import torch
    import paper_2604_08542_gb300 as ttt
    N = 4096
    g = torch.Generator(device="cuda").manual_seed(M + K)
    a = torch.randint(-4, 5, (M, K), generator=g, device="cuda").to(torch.bfloat16)
    b = torch.randint(-4, 5, (N, K), generator=g, device="cuda").to(torch.bfloat16)
    ref = (a.double() @ b.double().T).float()
    layer = ttt.TTT(1, 256, 256, dtype=torch.bfloat16)
    st = torch.cuda.current_stream().cuda_stream
    for fp32, acc in ((1, 0), (1, 1), (0, 0)):
        want = ref + 3.0 if acc else ref if fp32 else ref.to(torch.bfloat16)
        for _ in range(8):
            c = torch.full((M, N), 3.0, dtype=want.dtype, device="cuda")
            assert ttt.scal3r_ttt_gemm(layer.handle, a.data_ptr(), K, 1, b.data_ptr(), K, 1, c.data_ptr(), N, fp32,
                                       acc, M, N, K, None, 0, st) == 0
            assert torch.equal(c, want), (fp32, acc)
    assert layer.status() == 0
