"""The backward that takes dO in raster order and leaves a block-major copy on the way, against the one that is given the
copy: odd query counts, a strided dO, queries without a selected block."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer, lists_from_mask
from tests import _util as U

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, heads, nb, sb", [(1, 1, 1, 1), (1, 3, 3, 7), (2, 5, 4, 65), (1, 12, 2, 129)])
def test_copy_and_gradients(B, heads, nb, sb):
    shape = vb.make_shape(B, heads, 128, (nb, sb, 1), (1, sb, 1), "bf16")
    S = shape.S
    gen = torch.Generator().manual_seed(sb)
    mask = torch.rand(B * heads, S, nb, generator=gen) < 0.4
    mask[0, 0] = True
    kb_ptr, q_idx, q_ptr, q_pairs, n = lists_from_mask(mask.numpy())
    L = VmobaLayer(shape, n, with_backward=True)
    L.kb_ptr.copy_(kb_ptr); L.q_idx.copy_(q_idx); L.q_ptr.copy_(q_ptr); L.q_pairs.copy_(q_pairs)
    torch.manual_seed(sb)
    q, k, v = (torch.randn(B, S, heads, 128, device="cuda").bfloat16() for _ in range(3))
    do = torch.randn(B, S, heads, 256, device="cuda").bfloat16()[..., 64:192]
    L.partition_many((q, k, v), (L.q_bm, L.k_bm, L.v_bm), perm=L.perm)
    L.attn_fwd()
    L.partition(do, L.do_bm)
    want_do = L.do_bm.clone()
    want = [torch.full_like(q, 7.0) for _ in range(3)]
    L.attn_bwd_raster(None, *want)
    L.do_bm.fill_(7.0)
    got = [torch.full_like(q, 5.0) for _ in range(3)]
    L.attn_bwd_raster(do, *got, keep_do=True)
    L.check_status()
    assert torch.equal(L.do_bm, want_do)
    for name, a, b in zip(("dq", "dk", "dv"), got, want):        # sums taken in any order, rounded once
        U.assert_close(U.to_numpy_f32(a), U.to_numpy_f32(b), "bf16", name)
