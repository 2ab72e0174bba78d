"""The wide path's GEMMs at the edges of their tiles (GPU): 128 x 256 outputs on
one SM, 256 x 256 on a pair, K blocks of 64, the outputs staged through shared
memory or stored directly.

test_gemm_edges compares every float32 entry with the float64 product of the
same bfloat16 values: accumulation over up to 1,000 products is within 1000 *
2^-24 < 6e-5 of a row's sum of |a b|, which is below 16 times the largest entry
of these random sums: 16 * 6e-5 < 1e-3.  The bfloat16 output is the float32 one
rounded, to the bit.  The columns past N of the output's rows and the rows past
M keep their fill.  An operand given with its M values contiguous needs M to be a
multiple of 8 (its rows start on 16 bytes); others are refused.

test_layer_edges runs whole layers with chunks on both sides of 128 and 256
tokens, one or more heads, forward and backward, with the wide path's bar."""
import pytest

import oracle
from test_wide import _check, _check_grads, _fwd_bwd, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(8, 256, 8), (128, 1024, 64), (129, 1024, 72), (255, 4096, 128), (256, 512, 136),
                                   (257, 4096, 1000), (640, 2560, 200), (2600, 1024, 104)])
@pytest.mark.parametrize("a_kmajor,b_kmajor", [(1, 1), (1, 0), (0, 0), (0, 1)])
def test_gemm_edges(M, N, K, a_kmajor, b_kmajor):
    import torch
    import paper_2604_08542_gb300 as ttt
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16)
    B = torch.randn(N, K, generator=g).to(torch.bfloat16)
    ref = (A.double() @ B.double().T).cuda()
    pad = lambda n: (n + 7) // 8 * 8   # a row of an operand starts on 16 bytes
    def dev(x, kmajor):
        x = x if kmajor else x.T
        out = torch.zeros(x.shape[0], pad(x.shape[1]), dtype=torch.bfloat16, device="cuda")
        out[:, :x.shape[1]] = x.cuda()
        return out
    a, b = dev(A, a_kmajor), dev(B, b_kmajor)
    layer = ttt.TTT(1, 256, 256, dtype=torch.bfloat16)
    st = torch.cuda.current_stream().cuda_stream
    ldc, scale, fill = N + 8, ref.abs().max().item(), 3.0
    plain = None
    for fp32, acc in ((1, 0), (1, 1), (0, 0)):
        c = torch.full((M + 3, ldc), fill, dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
        rc = ttt.scal3r_ttt_gemm(layer.handle, a.data_ptr(), a.shape[1], a_kmajor, b.data_ptr(), b.shape[1], b_kmajor,
                                 c.data_ptr(), ldc, fp32, acc, M, N, K, None, 0, st)
        if not a_kmajor and M % 8:
            assert rc == ttt.SCAL3R_ERR_UNSUPPORTED
            continue
        assert rc == 0
        torch.cuda.synchronize()
        assert layer.status() == 0
        if fp32:
            err = (c[:M, :N].double() - (fill if acc else 0.0) - ref).abs().max().item() / scale
            assert err <= 1e-3, (acc, err)
            plain = c if not acc else plain
        else:
            assert torch.equal(c[:M, :N], plain[:M, :N].to(torch.bfloat16))
        assert (c[M:] == fill).all() and (c[:, N:] == fill).all()


@pytest.mark.parametrize("loss", ["dot", "mse"])
@pytest.mark.parametrize("H,D,F,lengths", [(2, 256, 512, [[255, 257], [1, 256]]), (1, 512, 1024, [[513, 127], [384]]),
                                           (1, 1024, 2048, [[1025, 129]])])
def test_layer_edges(H, D, F, lengths, loss):
    import torch
    import paper_2604_08542_gb300 as ttt
    layer = ttt.TTT(H, D, F, dtype=torch.bfloat16, loss=loss)
    _, lay, x, out = _run(H, D, F, lengths, seed=95, layer=layer)
    _check(out, oracle.forward(x["q"], x["k"], x["v"], x["lr"], x["w0"], lay, D, F, loss=loss, eps=1e-6))
    _, lay, x, grads = _fwd_bwd(H, D, F, lengths, seed=96, layer=layer)
    _check_grads(grads, oracle.backward(x["q"], x["k"], x["v"], x["lr"], x["w0"], lay, x["d_o"], D, F, loss=loss,
                                        eps=1e-6))
