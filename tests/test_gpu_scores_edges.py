"""The tensor-core scores at the edges of their tiles: query counts around a warp's 32 rows and a tile's 128, block counts
around the 32-column slabs, around the largest block range and with rows that are not multiples of 16 bytes."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb, sb", [(1, 31), (1, 700), (3, 11), (4, 8), (21, 6), (31, 33), (32, 4), (33, 4), (64, 5), (65, 2),
                                    (96, 3), (97, 4), (128, 3), (130, 1), (160, 4), (161, 2), (162, 3), (280, 3), (323, 1)])
@pytest.mark.parametrize("B, heads", [(1, 1), (2, 5)])
def test_scores_and_range(B, heads, nb, sb):
    shape = vb.make_shape(B, heads, 128, (nb, 1, sb), (1, 1, sb), "bf16")
    L = VmobaLayer(shape, 1024)
    torch.manual_seed(nb)
    L.q_bm.copy_(torch.randn(L.q_bm.shape, device="cuda"))
    L.k_bm.copy_(torch.randn(L.k_bm.shape, device="cuda"))
    guard = torch.full((L.scores.numel() + 512,), 7.0, device="cuda")
    L.scores = guard[256:-256].view(L.scores.shape)
    L.block_scores()
    L.check_status()
    assert torch.all(guard[:256] == 7.0) and torch.all(guard[-256:] == 7.0)
    q, c = L.q_bm.double(), L.centroids.double()
    # 384 exact products (three parts of every centroid value), added in fp32: at most 2^-23 of the sum of magnitudes each
    bound = 384 * 2.0 ** -23 * torch.matmul(q.abs(), c.abs().transpose(2, 3))
    assert torch.all((L.scores.double() - torch.matmul(q, c.transpose(2, 3))).abs() <= bound)
    flat = L.scores.view(B * heads, -1)
    assert torch.equal(L.score_range, torch.stack([flat.min(1).values, flat.max(1).values], 1))


@pytest.mark.parametrize("nb, sb", [(1, 31), (3, 11), (4, 8), (21, 6), (31, 33), (32, 5), (33, 7), (64, 5), (96, 3), (97, 6),
                                    (128, 3), (160, 7), (161, 3), (162, 3), (280, 3), (323, 5)])
def test_scores_carry_every_part_of_the_centroids(nb, sb):
    """A query with one non-zero channel, a power of two, has exact products: its scores are the fp32 centroid values times
    that power, whose three bf16 parts add up without rounding but for the accumulator's alignment (two units in the last
    place; the third part of a centroid lost would be 2^-17 of it)."""
    shape = vb.make_shape(1, 2, 128, (nb, 1, sb), (1, 1, sb), "bf16")
    L = VmobaLayer(shape, 1024)
    torch.manual_seed(nb + sb)
    L.k_bm.copy_(torch.randn(L.k_bm.shape, device="cuda"))
    channel = (torch.arange(shape.S, device="cuda") * 37) % 128
    L.q_bm.zero_()
    L.q_bm.scatter_(3, channel.view(1, 1, -1, 1).expand(1, 2, -1, 1), 4.0)
    L.block_scores()
    L.check_status()
    want = 4.0 * L.centroids.transpose(2, 3)[:, :, channel, :]                    # [1, heads, S, N_b]
    assert torch.all((L.scores - want).abs() <= 2.0 ** -22 * want.abs())
