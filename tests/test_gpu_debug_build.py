"""The range-checked build of the library (-DVMOBA_DEBUG, lib/libvmoba_debug.so): every index read from a work list
is checked before use and every workspace slice is followed by a guard zone that is verified after the stage's
kernels.  It stands in for a memory checker: the mid-size parity cases must run through it with the status word
clean, and a planted out-of-range list entry must be reported (and not followed: the access is redirected to
element 0, so nothing faults)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _debug_env():
    from paper_2506_23858_b200 import build
    return dict(os.environ, VMOBA_LIB=build.ensure_built(debug=True))


def test_mid_size_cases_run_clean_through_the_range_checked_build():
    r = subprocess.run([sys.executable, "-m", "pytest", "tests/test_gpu_layer.py", "tests/test_gpu_stages.py", "-m", "gpu",
                        "-q", "-x", "-p", "no:cacheprovider", "-k",
                        "mid_size or tails or select_matches or sparse_attention_forward_backward or raster or dense_attention"],
                       env=_debug_env(), cwd=ROOT, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-1000:]
    assert " passed" in r.stdout


PLANT = r"""
import numpy as np, torch
from paper_2506_23858_b200 import binding as vb, inputs as gen
from paper_2506_23858_b200.layer import VmobaLayer, default_capacity
w = gen.Workload("mid", 1, 2, 128, 6, 12, 26, (3, 6, 13), 0.25, "bf16", "smooth", 5)
data = gen.make_inputs(w, with_do=False)
shape = vb.shape_of(w)
L = VmobaLayer(shape, capacity=default_capacity(shape, w.tau))
dev = lambda n: torch.from_numpy(data[n + "_bits"].view(np.int16)).cuda().view(torch.bfloat16)
o = torch.empty_like(dev("q"))
L.forward(dev("q"), dev("k"), dev("v"), w.tau, o)
torch.cuda.synchronize()
print("clean", int(L.dev_status.item()))
L.q_idx[3] = w.S + 7            # a query position beyond the head
L.q_idx[11] = -2
L.attn_fwd()
torch.cuda.synchronize()
print("planted", int(L.dev_status.item()))
"""


def test_planted_out_of_range_entry_is_reported_by_the_range_checked_build():
    r = subprocess.run([sys.executable, "-c", PLANT], env=_debug_env(), cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    lines = dict(l.split() for l in r.stdout.strip().splitlines() if l.split()[0] in ("clean", "planted"))
    assert lines["clean"] == "0"
    assert lines["planted"] == "8"          # VMOBA_ERR_BOUNDS


CHAIN = r"""
import sys, torch
from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import SteppedAttention, VmobaLayer
out = []
for dtype, grid, block, heads, d in (("f32", (1, 8, 8), (1, 4, 4), 2, 64), ("bf16", (4, 16, 16), (2, 4, 8), 3, 128),
                                     ("bf16", (6, 12, 26), (3, 6, 13), 12, 128), ("bf16", (9, 32, 32), (3, 8, 16), 8, 128)):
    shape = vb.make_shape(1, heads, d, grid, block, dtype)
    L = VmobaLayer(shape, 4 * heads * shape.S, with_backward=True)
    gen = torch.Generator(device="cuda").manual_seed(3)
    sets = [[torch.randn(1, shape.S, heads, d, device="cuda", generator=gen).to(L.q_bm.dtype) for _ in range(4)] for _ in range(2)]
    for i in (0, 1, 0, 1):
        q, k, v, do = sets[i]
        o, dq, dk, dv, dense = (torch.empty_like(q) for _ in range(5))
        # (the head-wide top-k counts pairs where the threshold rule adds weights in any order: the same kernels, and the
        # same bits from run to run)
        L.partition_many((v, q, k), (L.v_bm, L.q_bm, L.k_bm), perm=L.perm)
        L.block_scores()
        L.select_rule(vb.SELECT_TOPK_GLOBAL, topk=2)
        L.attn_fwd()
        L.partition(o, L.o_bm, inverse=True)
        L.backward(do, dq, dk, dv)
        n = int(L.k_per_head.sum())
        out += [x.cpu() for x in (o, L.lse, dk, dv, L.mask_bits, L.kb_ptr, L.q_ptr, L.q_idx[:n], L.q_pairs[:n])]
        L.select_rule(vb.SELECT_TOPK_LOCAL, topk=3)
        SteppedAttention(L, 0.25, 1, 1.0).forward(0, q, k, v, dense)
        out += [L.mask_bits.cpu(), dense.cpu()]
    L.check_status()
torch.save(out, sys.argv[1])
"""


def test_overlapped_launches_give_what_serialised_ones_give(tmp_path):
    """The range-checked build launches every kernel after the end of the one before it; the library itself sets most of them
    up while that one still runs.  Forward, backward, selections and dense step over two sets of inputs in turn: bit for bit
    the same (dQ apart, whose parts come in any order)."""
    import torch
    for name, env in (("overlapped", dict(os.environ)), ("serialised", _debug_env())):
        r = subprocess.run([sys.executable, "-c", CHAIN, str(tmp_path / name)], env=env, cwd=ROOT, capture_output=True, text=True,
                           timeout=600)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    a, b = (torch.load(tmp_path / n) for n in ("overlapped", "serialised"))
    assert len(a) == len(b) and all(torch.equal(x, y) for x, y in zip(a, b))
