"""The row-update kernels of head_dim 64, hidden 128 (GPU) on both sides of
the rule that picks their form, and the squared-error loss's token rows.

A call with n chains updates 24 n blocks a step: up to 456 (19 chains on 152
SMs) they are resident together and take their slots six at a time, beyond
they take two at a time.  One chain of 2,500 tokens has the most slots, a
sequence without chunks only copies w0.  The first step's update, which forms
the row targets, is a form of its own.

Bars: the float32 path's 1e-5 normwise and, for the squared-error loss on the
bfloat16 path (its residual pieces and its token rows, 16 blocks a piece, at
chunks of 1 to 300 tokens), that path's 2e-2."""
import pytest

import ttt_synth as syn
from test_options_d64 import TOLS, _assert, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norm", ["row_w0", "unit", "none"])
@pytest.mark.parametrize("lengths,H,ckpt_every", [
    ([[2500, 130, 64]], 1, 1), ([[40, 33, 25]], 19, 1), ([[40, 33, 25]], 20, 1), ([[40, 33, 25], [], [17]], 8, 2),
    ([[40, 33], [], [17, 50]], 4, 1)])
def test_row_updates_fp32(lengths, H, ckpt_every, norm):
    errs, _ = _run("fp32", syn.layout_from_lengths(lengths), H, seed=91, norm=norm, ckpt_every=ckpt_every)
    _assert(errs, TOLS["fp32"])


@pytest.mark.parametrize("lengths,H", [([[1, 15, 16], [17, 2]], 2), ([[300, 129], [128, 127, 1]], 20)])
@pytest.mark.parametrize("ckpt_every", [1, 2])
def test_mse_token_rows_bf16(lengths, H, ckpt_every):
    errs, _ = _run("bf16", syn.layout_from_lengths(lengths), H, seed=92, loss="mse", ckpt_every=ckpt_every)
    _assert(errs, TOLS["bf16"])
