"""The float32 (64, 128) handle's schedule is the caller's (GPU): the tail fill it
reports is the one it runs, and without it scal3r_ttt_forward repeats the
allocation-free forward to the bit (both then cut the same pieces)."""
import pytest

import ttt_synth as syn
from _util import rel_inf, to_np, upload

pytestmark = pytest.mark.gpu


def test_tail_fill_of_a_float32_handle_is_obeyed():
    import torch
    import paper_2604_08542_gb300 as ttt
    H, D, F = 16, 64, 128
    lay = syn.layout_from_lengths([[2082, 2082], [2082, 2082]])   # 32 chains for 152 SMs: the fill pays
    g = upload(syn.make_inputs(lay.num_tokens, H, D, F, seed=12), torch.float32)
    layer = ttt.TTT(H, D, F, dtype=torch.float32)
    assert layer.schedule()["tail_fill"] == 3

    def forward():
        o, ck, wn, wf = layer.forward(g["q"], g["k"], g["v"], g["lr"], g["w0"], lay.chunk_offsets, lay.seq_chunk_ptr,
                                      want_final=True)
        return o, ck, wf

    def workspace_size():
        return ttt.scal3r_ttt_workspace_size(layer.handle, lay.chunk_offsets, lay.seq_chunk_ptr, False)

    filled, filled_size = forward(), workspace_size()
    layer.set_schedule(tail_fill=0)
    assert layer.schedule()["tail_fill"] == 0
    plain = forward()
    assert workspace_size() < filled_size   # one slot a piece: the fill's extra pieces are gone
    na = [torch.empty_like(t) for t in plain]
    cfg = ttt.scal3r_ttt_config(H, D, F, ttt.SCAL3R_FP32, ttt.SCAL3R_LOSS_DOT, ttt.SCAL3R_NORM_ROW_W0, 1e-6, 0)
    st = torch.cuda.current_stream().cuda_stream
    assert ttt.scal3r_ttt_forward_noalloc(cfg, *(g[n].data_ptr() for n in ("q", "k", "v", "lr", "w0")), 0,
                                          lay.chunk_offsets, lay.seq_chunk_ptr, na[0].data_ptr(), na[1].data_ptr(),
                                          None, na[2].data_ptr(), st) == 0
    for a, b, c in zip(plain, na, filled):
        assert torch.equal(a, b)
        assert rel_inf(to_np(c), to_np(a)) <= 1e-5
