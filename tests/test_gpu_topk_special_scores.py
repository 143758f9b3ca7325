"""Top-k per query on scores that float comparisons do not order, and some that they do: NaN, infinities, two zeros, rows of
equal scores.  A NaN has its place beyond the infinity of its sign, the two zeros are equal, ties go in block order, and every
query keeps exactly min(k, N_b) blocks."""
import numpy as np
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer
from tests import _util as U

pytestmark = pytest.mark.gpu


def _keys(scores):
    u = scores.view(np.uint32)
    u = np.where(u == 0x80000000, np.uint32(0), u)
    return np.where(u & 0x80000000, ~u, u | 0x80000000)


def _special(rng, heads, S, nb):
    x = rng.standard_normal((heads, S, nb)).astype(np.float32)
    pick = lambda p: rng.random(x.shape) < p
    rows = np.arange(S) % 12
    nan = np.float32(np.nan)
    neg_nan = np.uint32(0xffc00000).view(np.float32)
    x[:, rows == 1] = nan                                                      # a diverged query
    x[:, rows == 2, nb // 3] = nan                                             # one block
    x[:, rows == 3] = np.where(pick(0.4), nan, x)[:, rows == 3]
    x[:, rows == 4] = np.where(pick(0.4), neg_nan, x)[:, rows == 4]
    x[:, rows == 5] = np.where(pick(0.5), np.float32(np.inf), x)[:, rows == 5]
    x[:, rows == 6] = np.where(pick(0.9), np.float32(-np.inf), x)[:, rows == 6]
    x[:, rows == 7] = np.where(pick(0.5), np.float32(-0.0), np.float32(0.0))[:, rows == 7]
    x[:, rows == 8] = np.where(pick(0.8), np.where(pick(0.5), np.float32(-0.0), np.float32(0.0)), x)[:, rows == 8]
    x[:, rows == 9] = np.float32(1.5)
    x[:, rows == 10] = np.round(2 * x)[:, rows == 10]
    x[:, rows == 11] = np.where(pick(0.3), nan, np.where(pick(0.5), np.float32(np.inf), np.float32(-np.inf)))[:, rows == 11]
    return x


@pytest.mark.parametrize("nb", [3, 8, 20, 32, 33, 64, 65, 100, 161, 280, 1000])
def test_exactly_k_blocks_in_key_order(nb):
    heads, S = 3, 5 * nb * (1 if nb > 100 else 12)
    shape = vb.make_shape(1, heads, 64, (nb, S // nb, 1), (1, S // nb, 1), "f32")
    L = VmobaLayer(shape, heads * S * nb)
    x = _special(np.random.default_rng(nb), heads, S, nb)
    L.scores.copy_(torch.from_numpy(x).view(L.scores.shape))
    keys = _keys(x)
    order = np.argsort(-keys.astype(np.int64), axis=2, kind="stable")
    for k in sorted({1, 2, 5, min(9, nb), nb // 2, nb - 1, nb, nb + 3}):
        L.select_rule(vb.SELECT_TOPK_LOCAL, topk=k)
        L.check_status()
        kk = min(k, nb)
        want = np.zeros(x.shape, dtype=bool)
        np.put_along_axis(want, order[..., :kk], True, axis=2)
        assert np.array_equal(U.unpack_mask(L.mask_bits, heads, S, nb), want), k
        assert L.k_per_head.tolist() == [S * kk] * heads
        cutoff = np.where(want, keys, np.uint32(0xffffffff)).reshape(heads, -1).min(axis=1)
        assert np.array_equal(_keys(L.cutoff.cpu().numpy()), cutoff), k


@pytest.mark.parametrize("nb", [40, 140, 280])
def test_rows_unlike_the_one_before(nb):
    """The search starts from the threshold of the row before: rows of other scales, beyond and below it, and up to 1e38 away."""
    heads, S = 2, 24 * nb
    shape = vb.make_shape(1, heads, 64, (nb, S // nb, 1), (1, S // nb, 1), "f32")
    L = VmobaLayer(shape, heads * S * nb)
    rng = np.random.default_rng(nb)
    x = rng.standard_normal((heads, S, nb)).astype(np.float32)
    kind = rng.integers(0, 8, (heads, S, 1))
    size = np.float32(10.0) ** rng.integers(-30, 30, (heads, S, 1)).astype(np.float32)
    x = np.where(kind == 0, x * size, x)
    x = np.where(kind == 1, x + 1000 * rng.standard_normal((heads, S, 1)).astype(np.float32), x)
    x = np.where(kind == 2, np.where(np.arange(nb) == 3, np.float32(2.0), np.float32(1e-4) * x), x)
    x = np.where(kind == 3, np.float32(1e38) * np.sign(x), x)      # (ties)
    x = np.where(kind == 4, np.minimum(x, 0) - np.float32(1e38), x)
    x = np.where(kind == 5, np.where(np.arange(nb) % 3 == 0, np.float32(-np.inf), x), x).astype(np.float32)
    L.scores.copy_(torch.from_numpy(x).view(L.scores.shape))
    keys = _keys(x)
    order = np.argsort(-keys.astype(np.int64), axis=2, kind="stable")
    for k in (1, 2, 5, 9, nb // 2):
        L.select_rule(vb.SELECT_TOPK_LOCAL, topk=k)
        L.check_status()
        want = np.zeros(x.shape, dtype=bool)
        np.put_along_axis(want, order[..., :k], True, axis=2)
        assert np.array_equal(U.unpack_mask(L.mask_bits, heads, S, nb), want), k
