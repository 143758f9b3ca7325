"""Forwards on both sides of the sizes (1,024 lists; room for 4,096 items, which is capacity / 128 + lists + 1) up to which one
CTA writes the items' offsets and records, with lists of very different lengths: every query's result against plain softmax
attention over its blocks."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads, nb, sb, capacity", [(4, 256, 2, 300000), (4, 257, 2, 300000), (1, 8, 300, 8 * 2400),
                                                     (1, 8, 300, 4087 * 128), (1, 8, 300, 4088 * 128), (4, 40, 50, 3935 * 128),
                                                     (4, 40, 50, 3936 * 128), (1, 8, 300, 1 << 20), (2, 8, 400, 1 << 21)],
                         ids=["1024_lists", "1028_lists", "159_items", "4096_items", "4097_items", "narrow_4096_items",
                              "narrow_4097_items", "8201_items", "16401_items"])
def test_lists_of_any_length(heads, nb, sb, capacity):
    shape = vb.make_shape(1, heads, 128, (nb, sb, 1), (1, sb, 1), "bf16")
    S = shape.S
    L = VmobaLayer(shape, capacity)
    torch.manual_seed(nb)
    for buf in (L.q_bm, L.k_bm, L.v_bm):
        buf.normal_()
    scores = torch.randn(L.scores.shape, device="cuda") + torch.linspace(0.0, 3.0, nb, device="cuda")     # late blocks longer
    L.select(0.2, scores=scores)
    L.o_bm.fill_(7.0)
    L.attn_fwd()
    L.check_status()
    words = L.mask_bits.view(heads, S, -1)
    mask = ((words.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1).reshape(heads, S, -1)[:, :, :nb].bool()
    q, k, v = (x[0].float() for x in (L.q_bm, L.k_bm, L.v_bm))
    s = torch.matmul(q, k.transpose(1, 2)) * 128 ** -0.5
    s = s.masked_fill(~mask.repeat_interleave(sb, dim=2), float("-inf"))
    p = torch.nan_to_num(torch.softmax(s, dim=2), nan=0.0)            # no block: zero
    ref = torch.matmul(p, v)
    # weights and results rounded to bf16, partial rows to 2^-11 of their largest value: each at most 2^-8 of |v| <= 6
    assert float((L.o_bm[0].float() - ref).abs().max()) <= 2e-2
