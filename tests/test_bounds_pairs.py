"""The bounds-checking build launches the kernels of the ordinary one (GPU): the
same forward and backward of a wide layer, captured into a graph in one process
per build, has the same product launches (grid, block and shared memory: CTA pairs
and single CTAs differ in each), pairs among them.

A violation planted in a staged output (o registered 32 bytes short, see
test_bounds_build.py) is reported, and only the 16 outputs outside are left out."""
import ctypes
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class _KernelParams(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.c_void_p),
                ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _captured_launches(stream, fn):
    """[grid x y z, block x y z, shared bytes] of the kernels that fn() launches on `stream` (not run)."""
    cu = ctypes.CDLL("libcuda.so.1")
    st, graph, n = ctypes.c_void_p(stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(st, 2) == 0   # relaxed
    fn()
    assert cu.cuStreamEndCapture(st, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        kind, p = ctypes.c_int(), _KernelParams()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:   # a kernel
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
            out.append(list(p.dims))
    assert cu.cuGraphDestroy(graph) == 0
    return out


def _child():
    import torch
    import paper_2604_08542_gb300 as ttt
    import ttt_synth as syn
    from _util import upload
    H, D, F = 1, 512, 1024
    lay = syn.layout_from_lengths([[4000, 1300]])
    g = upload(syn.make_inputs(lay.num_tokens, H, D, F, seed=31, dtype="bf16", with_grad_out=True), torch.bfloat16)
    layer = ttt.TTT(H, D, F, dtype=torch.bfloat16)
    args = (g["q"], g["k"], g["v"], g["lr"], g["w0"], lay.chunk_offsets, lay.seq_chunk_ptr)
    ws = layer.workspace(lay.chunk_offsets, lay.seq_chunk_ptr, True, "cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        o, ck, wn, _ = layer.forward(*args)
        grads = layer.backward(*args, g["d_o"], ck, wn)
        torch.cuda.synchronize()

        def step():
            layer.forward(*args, workspace=ws, o=o, w_ckpt=ck, wnorm=wn)
            layer.backward(*args, g["d_o"], ck, wn, workspace=ws, out=grads)

        launches = _captured_launches(s.cuda_stream, step)
    planted = _planted() if ttt.LIB_PATH.endswith("_bounds.so") else None
    # 11 warps: the product kernel
    print(json.dumps({"library": ttt.LIB_PATH, "status": layer.status(),
                      "products": [d for d in launches if d[3] == 352], "planted": planted}))


def _planted():
    """o = h W2^T over hidden 4096 runs as a pair with staged outputs."""
    import torch
    import paper_2604_08542_gb300 as ttt
    import ttt_synth as syn
    from _util import upload
    H, D, F = 1, 256, 4096
    lay = syn.layout_from_lengths([[200]])
    g = upload(syn.make_inputs(lay.num_tokens, H, D, F, seed=32, dtype="bf16"), torch.bfloat16)
    layer = ttt.TTT(H, D, F, dtype=torch.bfloat16)
    args = (g["q"], g["k"], g["v"], g["lr"], g["w0"], lay.chunk_offsets, lay.seq_chunk_ptr)
    ref = layer.forward(*args)[0].reshape(-1)
    o = torch.full_like(g["q"], 7.0)
    ttt.scal3r_ttt_debug_bounds(layer.handle, 5, 32)   # o
    layer.forward(*args, o=o)
    torch.cuda.synchronize()
    flat = o.reshape(-1)
    return {"status": layer.status(), "tail_untouched": bool((flat[-16:] == 7.0).all()),
            "rest_written": bool(torch.equal(flat[:-16], ref[:-16]))}


@pytest.mark.gpu
def test_bounds_build_runs_the_same_product_kernels():
    from test_bounds_build import _bounds_lib
    from paper_2604_08542_gb300 import build as b
    path = os.pathsep.join([ROOT, os.path.join(ROOT, "tests"), os.environ.get("PYTHONPATH", "")])
    got = []
    for lib in (b.lib_path(), _bounds_lib()):
        r = subprocess.run([sys.executable, "-c", "import test_bounds_pairs as t; t._child()"], capture_output=True,
                           text=True, timeout=300, env=dict(os.environ, SCAL3R_TTT_LIBRARY=lib, PYTHONPATH=path))
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
        out = json.loads(r.stdout.strip().splitlines()[-1])
        assert out["library"] == lib and out["status"] == 0
        got.append(out["products"])
        planted = out["planted"]
    assert 230400 in {d[6] for d in got[0]}   # pairs: five 32 KB stages, 64 KB of staged outputs, 1 KB
    assert got[1] == got[0]
    assert planted == {"status": 9, "tail_untouched": True, "rest_written": True}   # SCAL3R_ERR_BOUNDS
