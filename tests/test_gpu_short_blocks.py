"""Forwards over key blocks of at most one 128-key tile, where a work item is over after a single tile and its roles hand
over to one another most often: many items per CTA, many passes, every pass the same bits and no wait that runs out."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sb, nb, heads, topk", [(128, 250, 12, 1), (128, 60, 12, 3), (96, 100, 4, 2), (16, 500, 4, 1), (2, 900, 2, 4)])
def test_many_short_items(sb, nb, heads, topk):
    shape = vb.make_shape(1, heads, 128, (nb, sb, 1), (1, sb, 1), "bf16")
    L = VmobaLayer(shape, heads * shape.S * topk, with_backward=True)
    torch.manual_seed(sb)
    for buf in (L.q_bm, L.k_bm, L.v_bm, L.scores):
        buf.normal_()
    L.select_rule(vb.SELECT_TOPK_LOCAL, topk=topk)
    want = None
    for _ in range(60):
        L.attn_fwd()
        got = (L.o_bm.clone(), L.o_resid.clone(), L.lse.clone())
        want = want or got
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    L.check_status()
    # the last head against plain softmax attention over the chosen blocks (see test_gpu_item_records for the bound)
    S = shape.S
    words = L.mask_bits.view(heads, S, -1)[-1]
    mask = ((words.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(S, -1)[:, :nb].bool()
    q, k, v = (x[0, -1].float() for x in (L.q_bm, L.k_bm, L.v_bm))
    for i in range(0, S, 4096):
        s = (q[i:i + 4096] @ k.T) * 128 ** -0.5
        s = s.masked_fill(~mask[i:i + 4096].repeat_interleave(sb, dim=1), float("-inf"))
        assert float((L.o_bm[0, -1, i:i + 4096].float() - torch.softmax(s, dim=1) @ v).abs().max()) <= 2e-2
