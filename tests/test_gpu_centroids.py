"""Block means for every type and head dimension, with as many blocks as are still summed by four CTAs each and with
more, and with block sizes around the rows that a thread has in flight."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sb", [1, 7, 8, 255, 256, 257])
@pytest.mark.parametrize("heads, nb", [(3, 5), (8, 73), (8, 75)], ids=["15_blocks", "584_blocks", "600_blocks"])
@pytest.mark.parametrize("dtype, d", [("f32", 64), ("f32", 128), ("bf16", 64), ("bf16", 128)])
def test_block_means(dtype, d, heads, nb, sb):
    shape = vb.make_shape(1, heads, d, (nb, 1, sb), (1, 1, sb), dtype)
    L = VmobaLayer(shape, 1024)
    torch.manual_seed(11)
    L.q_bm.zero_()
    L.k_bm.copy_(torch.randn(L.k_bm.shape, device="cuda"))
    L.centroids.fill_(7.0)
    L.block_scores()
    L.check_status()
    k = L.k_bm.double().view(1, heads, nb, sb, d)
    # sums of at most sb fp32 additions and one rounded product: each rounds by at most 2^-24 of the sum of magnitudes
    bound = (sb + 2) * 2.0 ** -24 * k.abs().mean(3)
    assert torch.all((L.centroids.double() - k.mean(3)).abs() <= bound)
