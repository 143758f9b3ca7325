"""A layer's kernels overlap their launches with the kernel before them: passes over alternating inputs in the same
buffers, enqueued without a pause, give what the same passes give with a synchronisation after every stage.  The sizes
lie on both sides of the tensor size (16 MB) up to which the long kernels take part."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer, default_capacity
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype, grid, block, heads, d", [
    ("f32", (1, 8, 8), (1, 4, 4), 2, 64), ("bf16", (4, 16, 16), (2, 4, 8), 3, 128),
    ("bf16", (8, 32, 32), (2, 8, 16), 8, 128), ("bf16", (9, 32, 32), (3, 8, 16), 8, 128)],
    ids=["tiny", "small", "16MB", "18MB"])
def test_overlapped_passes_match_synchronised_ones(dtype, grid, block, heads, d):
    shape = vb.make_shape(1, heads, d, grid, block, dtype)
    L = VmobaLayer(shape, default_capacity(shape, 0.25), with_backward=True)
    torch.manual_seed(3)
    sets = [[torch.randn(1, shape.S, heads, d, device="cuda").to(L.q_bm.dtype) for _ in range(4)] for _ in range(2)]

    def one(i, sync):
        q, k, v, do = sets[i]
        outs = [torch.empty_like(q) for _ in range(4)]
        pause = torch.cuda.synchronize if sync else (lambda: None)
        L.partition(q, L.q_bm, perm=L.perm); pause()
        L.partition(k, L.k_bm); pause()
        L.partition(v, L.v_bm); pause()
        L.block_scores(); pause()
        L.select(0.25); pause()
        L.attn_fwd(); pause()
        L.partition(outs[0], L.o_bm, inverse=True); pause()
        L.backward(do, *outs[1:]); pause()
        return outs + [L.mask_bits.clone(), L.lse.clone()]

    want = [one(i, True) for i in (0, 1)]
    got = [one(i, False) for i in (0, 1, 0)]
    L.check_status()
    for i, g in zip((0, 1, 0), got):
        for n in (0, 4, 5):
            assert torch.equal(g[n], want[i][n])
        for n, name in ((1, "dq"), (2, "dk"), (3, "dv")):      # the parts of a gradient are added in any order
            U.assert_close(U.to_numpy_f32(g[n]), U.to_numpy_f32(want[i][n]), dtype, name)
