"""The register-tiled float32 kernels (head_dim 64, hidden 128) at the edges of
their token tiles (16, 32 and 64 tokens) and under the planner's tail fill,
against the FP64 oracle (GPU).  With more chains than SMs every task is one
piece, so a chunk of n tokens runs its full tiles and its remainder in one CTA.

Bar: the float32 path's, max|x - ref| / max|ref| <= 1e-5 for every output and gradient."""
import numpy as np
import pytest

import oracle
import ttt_synth as syn
from _util import rel_inf, to_np, upload

pytestmark = pytest.mark.gpu

TOL = 1e-5
EDGES = [[16, 17], [31, 1], [32, 33], [63, 64, 65], [15, 81, 48]]


@pytest.mark.parametrize("loss,per_matrix,lengths,H", [
    ("dot", False, EDGES, 32), ("dot", True, EDGES, 32), ("mse", False, EDGES, 32), ("mse", True, EDGES, 32),
    ("dot", False, [[1500, 700]], 16), ("mse", True, [[900, 333], [640]], 9)])
def test_fp32_tile_edges_and_fill(loss, per_matrix, lengths, H):
    import torch
    import paper_2604_08542_gb300 as ttt
    D, F = 64, 128
    lay = syn.layout_from_lengths(lengths)
    T = lay.num_tokens
    x = syn.make_inputs(T, H, D, F, seed=71, with_grad_out=True)
    if per_matrix:
        x["lr"] = syn.per_matrix_lr(71, T, H)
    g = upload(x, torch.float32)
    layer = ttt.TTT(H, D, F, dtype=torch.float32, loss=loss, lr_per_matrix=per_matrix)
    args = (g["q"], g["k"], g["v"], g["lr"], g["w0"], lay.chunk_offsets, lay.seq_chunk_ptr)
    o, ck, wn, wf = layer.forward(*args, want_final=True)
    grads = layer.backward(*args, g["d_o"], ck, wn)
    torch.cuda.synchronize()
    assert layer.status() == 0
    oargs = (x["q"], x["k"], x["v"], x["lr"], x["w0"], lay)
    ref = oracle.forward(*oargs, D, F, loss=loss, eps=1e-6)
    ref.update(oracle.backward(*oargs, x["d_o"], D, F, loss=loss, eps=1e-6))
    got = {"o": o, "w_ckpt": ck, "wnorm": wn, "w_final": wf, **dict(zip(("dq", "dk", "dv", "dlr", "dw0"), grads))}
    errs = {n: rel_inf(to_np(t), np.asarray(ref[n])) for n, t in got.items()}
    bad = {n: e for n, e in errs.items() if not e <= TOL}
    assert not bad, f"errors above {TOL}: {bad} (all: {errs})"
