"""The selection's lists against the mask they come from, around the sizes at which its prefix sums change shape: one or
several segments per thread, one or several groups of 32 blocks, one or several trips of the scans (8,192 elements); and
scores that crowd into one histogram bin, with room for the candidates in a CTA's buffer and without."""
import numpy as np
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer

pytestmark = pytest.mark.gpu


def _mask(L):
    words = L.mask_bits.view(L.BH, L.S, -1)
    bits = (words.unsqueeze(-1) >> torch.arange(32, device="cuda", dtype=torch.int32)) & 1
    return bits.reshape(L.BH, L.S, -1)[:, :, :L.Nb].bool()


def _check_lists(L):
    mask = _mask(L)
    by_block = mask.transpose(1, 2)
    n = int(mask.sum())
    ids = torch.zeros(by_block.shape, dtype=torch.int32, device="cuda")
    ids[by_block] = torch.arange(n, dtype=torch.int32, device="cuda")
    ends = lambda m: torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), m.sum(-1).flatten().cumsum(0)])
    assert torch.equal(L.kb_ptr.long(), ends(by_block))
    assert torch.equal(L.q_ptr.long(), ends(mask))
    assert torch.equal(L.q_idx[:n].long(), by_block.nonzero()[:, 2])
    assert torch.equal(L.q_pairs[:n], ids.transpose(1, 2)[mask])
    assert torch.equal(L.k_per_head, mask.sum((1, 2)))
    return n


@pytest.mark.parametrize("heads, S, nb", [(1, 8, 1), (3, 512, 2), (2, 513, 32), (5, 16384, 32), (2, 16896, 33),
                                          (129, 64, 64), (33, 260, 260), (1, 40000, 80)])
def test_lists_match_the_mask(heads, S, nb):
    shape = vb.make_shape(1, heads, 128, (nb, 1, S // nb), (1, 1, S // nb), "bf16")
    L = VmobaLayer(shape, heads * shape.S * max(1, nb // 4) + 4096)
    torch.manual_seed(S)
    L.select(0.1, scores=torch.randn(L.scores.shape, device="cuda"))
    L.check_status()
    assert _check_lists(L) > 0


@pytest.mark.parametrize("heads, S, nb", [(2, 2048, 1024), (2, 2050, 1025), (1, 4098, 2049), (1, 8192, 8192)])
def test_lists_of_short_segments(heads, S, nb):
    """So many blocks that a segment has fewer than 128 queries (from 1,025 on; 32 from 2,049 on): more threads than queries."""
    shape = vb.make_shape(1, heads, 64, (nb, 1, S // nb), (1, 1, S // nb), "f32")
    L = VmobaLayer(shape, heads * S * 64)
    torch.manual_seed(nb)
    for _ in range(2):
        L.select_rule(vb.SELECT_TOPK_GLOBAL, topk=17, scores=torch.randn(L.scores.shape, device="cuda"))
        L.check_status()
        assert _check_lists(L) == heads * S * 17


@pytest.mark.parametrize("spread", [1.0, 1e-2, 1e-4], ids=["spread", "few_bins", "one_bin"])
def test_crowded_bins(spread):
    shape = vb.make_shape(1, 2, 128, (64, 1, 64), (1, 1, 64), "bf16")
    L = VmobaLayer(shape, 2 * shape.S * 64)
    torch.manual_seed(7)
    scores = spread * torch.randn(L.scores.shape, device="cuda")
    scores[..., 0, 0], scores[..., 0, 1] = 40.0, -40.0           # the histogram's range
    L.select(0.3, scores=scores)
    L.check_status()
    _check_lists(L)
    for h in range(2):
        s = np.sort(scores[0, h].double().cpu().numpy().ravel())[::-1]
        w = np.exp((s - s[0]) * 128 ** -0.5)
        mass = np.cumsum(w)
        k = int(L.k_per_head[h])
        # the shortest prefix of the sorted pairs that reaches the share; a CTA adds the weights of its share of the pairs
        # (P over at least 32 CTAs) in fp32, each addition off by at most 2^-24 of the sum
        eps = 2.0 ** -24 * s.size / 32
        assert mass[k - 1] >= 0.3 * mass[-1] * (1 - eps) and (k == 1 or mass[k - 2] <= 0.3 * mass[-1] * (1 + eps))
