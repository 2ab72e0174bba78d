"""The wide path's product when every CTA pair takes several output tiles and the
last row block leaves warps without rows (GPU): 65 row blocks of 256 by 16 column
blocks for 76 pairs, the last block with 16 or 128 of its rows.  At K of one or two
steps the launch is bound by its stores and a tile's staging buffers are still
being read when the next tile's accumulator is ready; a bfloat16 output is staged
from K = 768 on only (see below).

The operands are whole numbers up to 4 and K <= 1000: every sum is below 2^24, so
float32 holds it exactly in any order and the outputs are compared to the bit
(the bfloat16 one is the rounded sum).

test_short_bf16_products_run_as_single_ctas checks the form a product takes: pairs
cost a short one with a bfloat16 output up to a third more time."""
import pytest

from test_bounds_pairs import _captured_launches

pytestmark = pytest.mark.gpu

SINGLE, PAIR = 197632, 230400   # bytes of shared memory of the two forms


@pytest.mark.parametrize("M,K", [(16400, 64), (16400, 128), (16512, 64), (16400, 768), (16512, 1000)])
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


@pytest.mark.parametrize("M,N,K,fp32,form", [
    (130, 256, 64, 0, SINGLE), (5000, 1024, 64, 0, SINGLE), (16656, 4096, 512, 0, SINGLE), (2082, 1024, 2048, 0, SINGLE),
    (8328, 1024, 2048, 0, PAIR), (16656, 2048, 768, 0, PAIR), (50000, 256, 1024, 0, PAIR), (5000, 1024, 64, 1, PAIR)])
def test_short_bf16_products_run_as_single_ctas(M, N, K, fp32, form):
    import torch
    import paper_2604_08542_gb300 as ttt
    a = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    b = torch.zeros((N, K), dtype=torch.bfloat16, device="cuda")
    c = torch.zeros((M, N), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
    layer = ttt.TTT(1, 256, 256, dtype=torch.bfloat16)
    s = torch.cuda.Stream()

    def product():
        assert ttt.scal3r_ttt_gemm(layer.handle, a.data_ptr(), K, 1, b.data_ptr(), K, 1, c.data_ptr(), N, fp32, 0, M,
                                   N, K, None, 0, s.cuda_stream) == 0

    assert [d[6] for d in _captured_launches(s.cuda_stream, product)] == [form]
