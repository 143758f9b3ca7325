"""A layer's forward and backward captured into a CUDA graph: replayed over new contents of the captured buffers they give what
eager calls give.  The fp32 path has a memset among its kernels; the last size lies above the tensor size (16 MB) up to which
the long kernels are launched ahead of the end of the one before them."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype, grid, block, heads, d", [
    ("f32", (1, 8, 8), (1, 4, 4), 2, 64), ("bf16", (6, 12, 26), (3, 6, 13), 2, 128), ("bf16", (9, 32, 32), (3, 8, 16), 8, 128)],
    ids=["f32", "small", "18MB"])
def test_captured_layer_matches_eager(dtype, grid, block, heads, d):
    shape = vb.make_shape(1, heads, d, grid, block, dtype)
    L = VmobaLayer(shape, 4 * heads * shape.S, with_backward=True)
    torch.manual_seed(5)
    sets = [[torch.randn(1, shape.S, heads, d, device="cuda").to(L.q_bm.dtype) for _ in range(4)] for _ in range(3)]
    ins = [x.clone() for x in sets[0]]
    outs = [torch.empty_like(ins[0]) for _ in range(4)]

    def layer():
        # forward() with the head-wide top-k in the place of the threshold rule: the same kernels, but they count pairs where
        # the other adds weights in any order, so that the selection is the same from run to run
        q, k, v, do = ins
        L.partition_many((v, q, k), (L.v_bm, L.q_bm, L.k_bm), perm=L.perm)
        L.block_scores()
        L.select_rule(vb.SELECT_TOPK_GLOBAL, topk=2)
        L.attn_fwd()
        L.partition(outs[0], L.o_bm, inverse=True)
        L.backward(do, *outs[1:])

    def results():
        return [x.clone() for x in outs] + [L.mask_bits.clone(), L.lse.clone()]

    want = []
    for s in sets:
        for x, y in zip(ins, s):
            x.copy_(y)
        layer()
        want.append(results())
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        layer()
    for i in (2, 0, 1, 1, 2):
        for x, y in zip(ins, sets[i]):
            x.copy_(y)
        graph.replay()
        got = results()
        for n in (0, 2, 3, 4, 5):
            assert torch.equal(got[n], want[i][n])
        U.assert_close(U.to_numpy_f32(got[1]), U.to_numpy_f32(want[i][1]), dtype, "dq")     # its parts are added in any order
    L.check_status()
