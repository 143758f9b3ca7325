"""The tensor-core kernels at the edges of their tiles: hand-built lists on the edges of the forward's 256-row items and
the backward's 128-query units, against key blocks of three tiles and more (the forward's two-tile kernel) whose last
tile holds one key, is full or in between; and the dense path at sequence lengths around its tiles."""
import numpy as np
import pytest
import torch

from oracle import vmoba_oracle as orc
from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200 import inputs as gen
from paper_2506_23858_b200.layer import VmobaLayer, lists_from_mask
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("raster", [False, True], ids=["block_major", "raster"])
@pytest.mark.parametrize("keys", [257, 300, 384, 513])
def test_lists_on_item_and_unit_edges(keys, raster):
    w = gen.Workload("tiles", 1, 1, 128, 12, keys, 1, (1, keys, 1), 0.25, "bf16", "smooth", 19)
    data = gen.make_inputs(w)
    perm, _ = orc.partition_perm(w.T, w.H, w.W, *w.block)
    q, k, v, do = (data[n][0, :, 0][perm] for n in ("q", "k", "v", "do"))
    rng = np.random.default_rng(4)
    counts = [0, 1, 16, 127, 128, 129, 255, 256, 257, 384, 385, 600]
    mask = np.zeros((1, w.S, w.n_blocks), dtype=bool)
    for j, c in enumerate(counts):
        mask[0, rng.choice(w.S // 2, size=c, replace=False), j] = True      # half of the queries have no block
    kb_ptr, q_idx, q_ptr, q_pairs, n = lists_from_mask(mask)
    L = VmobaLayer(vb.shape_of(w), capacity=n, with_backward=True)
    dev = lambda name: U.to_device(w, data, name)
    for name, buf in (("q", L.q_bm), ("k", L.k_bm), ("v", L.v_bm), ("do", L.do_bm)):
        buf.copy_(U.bm_to_device(w, U.block_major(w, data, name, perm)))
    L.kb_ptr.copy_(kb_ptr); L.q_idx.copy_(q_idx); L.q_ptr.copy_(q_ptr); L.q_pairs.copy_(q_pairs)
    if raster:
        L.partition(dev("q"), L.q_bm, perm=L.perm)
        o, dq, dk, dv = (torch.full_like(dev("q"), 7.0) for _ in range(4))
        L.attn_fwd_raster(o)
        L.attn_bwd_raster(dev("do"), dq, dk, dv)
        o, dq, dk, dv = (U.to_numpy_f32(t)[0, :, 0][perm] for t in (o, dq, dk, dv))
    else:
        L.o_bm.fill_(7.0)
        L.attn_fwd()
        L.attn_bwd()
        o, dq, dk, dv = (U.to_numpy_f32(t).reshape(w.S, w.head_dim) for t in (L.o_bm, L.dq_bm, L.dk_bm, L.dv_bm))
    L.check_status()
    scale = w.head_dim ** -0.5
    o_ref, lse_ref = orc.sparse_attn_fwd(q, k, v, mask[0], scale)
    dq_ref, dk_ref, dv_ref = orc.sparse_attn_bwd(q, k, v, mask[0], scale, do)
    lse = L.lse.cpu().numpy().reshape(w.S)
    empty = ~mask[0].any(axis=1)
    assert np.all(o[empty] == 0) and np.all(np.isneginf(lse[empty])) and np.all(dq[empty] == 0)
    assert U.max_abs(lse[~empty], lse_ref[~empty]) <= 2e-2
    for name, got, ref in (("o", o, o_ref), ("dq", dq, dq_ref), ("dk", dk, dk_ref), ("dv", dv, dv_ref)):
        U.assert_close(got, ref, w.dtype, name)


@pytest.mark.parametrize("S", [1, 64, 127, 128, 129, 257, 400])
def test_dense_around_tiles(S):
    w = gen.Workload("dense_tiles", 1, 2, 128, 1, S, 1, (1, S, 1), 1.0, "bf16", "smooth", 23)
    data = gen.make_inputs(w)
    q, k, v, do = (U.to_device(w, data, n).permute(0, 2, 1, 3).contiguous() for n in ("q", "k", "v", "do"))
    shape = vb.shape_of(w)
    o, dq, dk, dv = (torch.full_like(q, 7.0) for _ in range(4))
    lse = torch.empty(w.heads * S, dtype=torch.float32, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(vb.workspace_bytes(shape, vb.STAGE_FULL_BWD), dtype=torch.uint8, device="cuda")
    vb.vmoba_full_attn(shape, q, k, v, o, lse, do, dq, dk, dv, st, ws)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    scale = w.head_dim ** -0.5
    for h in range(w.heads):
        qh, kh, vh, dh = (data[n][0, :, h] for n in ("q", "k", "v", "do"))
        o_ref, lse_ref = orc.dense_attn_fwd(qh, kh, vh, scale)
        grads = orc.dense_attn_bwd(qh, kh, vh, scale, dh)
        U.assert_close(U.to_numpy_f32(o[0, h]), o_ref, w.dtype, "o")
        assert U.max_abs(lse.view(w.heads, S)[h].cpu().numpy(), lse_ref) <= 2e-2
        for name, got, ref in zip(("dq", "dk", "dv"), (dq, dk, dv), grads):
            if S > 1 or name == "dv":       # a single key: the gradients of q and k vanish, rounding is all there is
                U.assert_close(U.to_numpy_f32(got[0, h]), ref, w.dtype, name)
