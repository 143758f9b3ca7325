"""The two routes to a head's cutoff: small pools go through one kernel, a cluster per head, larger ones through histograms of the
matrix.  A pool of m copies of the same scores has m times the mass above any score, so the cutoff is the same on both and every copy
keeps the same pairs."""
import math

import numpy as np
import pytest
import torch

from paper_2506_23858_b200 import binding as vb

pytestmark = pytest.mark.gpu
POOL_MAX = 1 << 20          # beyond every pool that the cluster kernel takes


def _run(shape, scores, rule, tau=0.25, topk=1, score_range=None, capacity=None):
    BH, S, Nb = shape.B * shape.heads, shape.S, shape.n_blocks
    cap = capacity or BH * S * Nb
    new = lambda n, dt=torch.int32: torch.full((n,), -7, dtype=dt, device="cuda")
    out = dict(mask=new(BH * S * shape.mask_words), kb_ptr=new(BH * Nb + 1), q_idx=new(cap), q_ptr=new(BH * S + 1), q_pairs=new(cap),
               k=new(BH, torch.int64), cutoff=torch.full((BH,), float("nan"), device="cuda"),
               status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    ws = torch.full((vb.workspace_bytes(shape, vb.STAGE_SELECT, cap),), 0x5a, dtype=torch.uint8, device="cuda")
    args = (out["mask"], out["kb_ptr"], out["q_idx"], out["q_ptr"], out["q_pairs"], cap, out["k"], out["cutoff"], out["status"], ws)
    if score_range is None:
        vb.vmoba_select_rule_apply(shape, scores, rule, tau, topk, *args)
    else:
        vb.vmoba_select_ranged(shape, scores, score_range, rule, tau, topk, *args)
    torch.cuda.synchronize()
    return out


def _mask(shape, out):
    BH, S, Nb = shape.B * shape.heads, shape.S, shape.n_blocks
    w = out["mask"].cpu().numpy().view(np.uint32).reshape(BH, S, -1)
    bits = ((w[..., None] >> np.arange(32, dtype=np.uint32)) & 1).astype(bool).reshape(BH, S, -1)
    assert not bits[..., Nb:].any()
    return bits[..., :Nb]


def _check_lists(shape, out, m):
    """kb_ptr, q_idx, q_ptr, q_pairs and the counts are those of the mask."""
    BH, S, Nb = m.shape
    assert out["k"].tolist() == m.sum((1, 2)).tolist()
    per_block = m.sum(1).reshape(-1)
    assert out["kb_ptr"].tolist() == [0] + np.cumsum(per_block).tolist()
    assert out["q_ptr"].tolist() == [0] + np.cumsum(m.sum(2).reshape(-1)).tolist()
    n = int(m.sum())
    bh, j, q = np.nonzero(m.transpose(0, 2, 1))          # by block, then query
    assert np.array_equal(out["q_idx"][:n].cpu().numpy(), q)
    place = np.zeros(m.shape, dtype=np.int64)
    place[bh, q, j] = np.arange(n)
    assert np.array_equal(out["q_pairs"][:n].cpu().numpy(), place[m])


def _copies(small):
    """The shape with further query rows that makes the pool larger than POOL_MAX: the same blocks per row, `copies` times the frames
    and the frames per block."""
    copies = POOL_MAX // (small.S * small.n_blocks) + 1
    big = _shape(small.heads, (small.T * copies, small.H, small.W), (small.bT * copies, small.bH, small.bW))
    assert big.n_blocks == small.n_blocks and big.S * big.n_blocks > POOL_MAX
    return copies, big


def _repeat(x, copies):
    heads, S, Nb = x.shape
    return x[:, None].expand(heads, copies, S, Nb).reshape(heads, copies * S, Nb).contiguous()


def _shape(heads, grid, block):
    return vb.make_shape(1, heads, 64, grid, block, "f32")


# grid, block: one CTA; several, some of them without a segment; rows of an odd number of blocks (slices off 16-byte boundaries); short
# rows; rows of several mask words; up to the largest slices that shared memory holds (319,488 scores in eight CTAs)
SHAPES = [((1, 7, 9), (1, 1, 1)), ((4, 8, 8), (1, 8, 8)), ((3, 43, 8), (3, 43, 1)), ((5, 13, 11), (1, 13, 11)), ((2, 33, 37), (1, 3, 37)),
          ((8, 24, 35), (2, 3, 35)), ((7, 40, 35), (7, 10, 5)), ((20, 17, 6), (1, 17, 1)), ((8, 24, 52), (2, 6, 26))]


@pytest.mark.parametrize("grid,block", SHAPES)
@pytest.mark.parametrize("rule,tau,topk", [(vb.SELECT_THRESHOLD_GLOBAL, 0.25, 0), (vb.SELECT_THRESHOLD_GLOBAL, 1.0, 0),
                                           (vb.SELECT_TOPK_GLOBAL, 0.0, 3)])
def test_pool_kernel_agrees_with_the_passes_over_the_matrix(grid, block, rule, tau, topk):
    heads = 3
    small = _shape(heads, grid, block)
    S, Nb = small.S, small.n_blocks
    copies, large = _copies(small)
    g = torch.Generator(device="cuda").manual_seed(S * Nb)
    x = 4.0 * torch.randn((heads, S, Nb), generator=g, device="cuda")
    before = vb.kernel_launches()
    a = _run(small, x, rule, tau, topk)
    ranged = _run(small, x, rule, tau, topk, score_range=torch.stack([x.amin((1, 2)), x.amax((1, 2))], 1).contiguous())
    assert vb.kernel_launches() - before == 4                  # the two kernels of the small route, twice
    b = _run(large, _repeat(x, copies), rule, tau, topk, capacity=int(heads * large.S * Nb))
    ma = _mask(small, a)
    for out in (a, ranged):
        _check_lists(small, out, _mask(small, out))
        assert int(out["status"]) == 0
    # the budget of the pair-count rule and, for masses, one pair at the cutoff: sums of millions of fp32 weights in any order
    # are off by 1e-6 of the whole, less than a pair's weight at most cutoffs
    mb = _mask(large, b).reshape(heads, copies, S, Nb)
    for other in (_mask(small, ranged), mb[:, 0], mb[:, -1]):
        assert (np.abs(other.sum((1, 2)) - ma.sum((1, 2))) <= (1 if rule == vb.SELECT_THRESHOLD_GLOBAL else 0)).all()
        assert (other != ma).sum() <= heads
    assert torch.allclose(a["cutoff"], b["cutoff"], atol=1e-2)


@pytest.mark.parametrize("tau", [0.02, 0.25, 0.9])
@pytest.mark.parametrize("values", ["flat", "sharp", "few hold the mass", "outlier", "one side"])
# 63,600 queries x 80 blocks (ten million scores in all: the passes), and small pools of one, four and eight CTAs
@pytest.mark.parametrize("grid,block", [((12, 100, 53), (3, 5, 53)), ((4, 13, 11), (1, 13, 11)), ((6, 12, 26), (3, 6, 13)), ((8, 24, 35), (2, 3, 35))])
def test_cutoff_against_a_sort(grid, block, values, tau):
    """Both routes find the cutoff whatever the scores look like: against a sort in 64 bits.  The sums of 3 million fp32 weights are
    off by 1e-6 of the whole, those of the small route (up to 112 per thread) by no more."""
    shape = _shape(2, grid, block)
    heads, S, Nb = shape.heads, shape.S, shape.n_blocks
    g = torch.Generator(device="cuda").manual_seed(7)
    x = torch.randn((heads, S, Nb), generator=g, device="cuda")
    if values == "flat":
        x *= 0.05
    elif values == "sharp":
        x *= 20.0
    elif values == "few hold the mass":
        x *= 45.0
    elif values == "outlier":
        x[:, S // 3, Nb // 2] = 60.0
        x[:, S // 4, 0] = -5e3
    else:
        x = -torch.exp(x)
    out = _run(shape, x, vb.SELECT_THRESHOLD_GLOBAL, tau, score_range=torch.stack([x.amin((1, 2)), x.amax((1, 2))], 1).contiguous())
    for h in range(heads):
        v = x[h].flatten().double().sort(descending=True).values
        cs = torch.exp((v - v[0]) / 8.0).cumsum(0)                                  # scale 64 ** -0.5
        want = min(int((cs < tau * cs[-1]).sum()), v.numel() - 1)                   # index of the pair that reaches the target
        k = int((x[h] >= out["cutoff"][h]).sum())
        assert k == int(out["k"][h])
        assert abs(float(cs[k - 1] - cs[want])) <= 2e-6 * float(cs[-1]), (h, k, want)
    assert int(out["status"]) == 0


def test_last_candidates_of_a_small_pool_are_added_up_in_64_bits():
    """One pair of weight 1, 30 of 2^-25 and one of 2^-26, all among the last candidates: which of the small ones reaches the target
    does not show in fp32, where 1 + 2^-25 is 1.  (A candidate per warp lane, so that the mass of the pool is exact.)"""
    heads = 8
    shape = _shape(heads, (4, 64, 1), (1, 64, 1))
    S, Nb = shape.S, shape.n_blocks
    per_unit = 0.125 * math.log2(math.e)                       # octaves of weight per unit of score: scale 64 ** -0.5
    x = torch.linspace(-2e6, -1.9e6, S * Nb, dtype=torch.float64)
    x[0] = 0.0
    for j in range(30):
        x[1 + j] = -25.0 / per_unit * (1 + j * 2.0 ** -20)
    x[31] = -26.0 / per_unit
    x = x.float().reshape(1, S, Nb).expand(heads, S, Nb).contiguous().cuda()
    v = x[0].flatten().double().sort(descending=True).values
    cs = torch.exp(v / 8.0).cumsum(0)
    for m in range(1, 15):
        tau = 1.0 - m * 2.0 ** -24
        out = _run(shape, x, vb.SELECT_THRESHOLD_GLOBAL, tau)
        assert out["k"].tolist() == [int((cs < tau * cs[-1]).sum()) + 1] * heads, m


@pytest.mark.parametrize("values", ["constant", "zeros", "two", "infinite", "nan"])
@pytest.mark.parametrize("rule,tau,topk", [(vb.SELECT_THRESHOLD_GLOBAL, 0.3, 0), (vb.SELECT_TOPK_GLOBAL, 0.0, 2)])
def test_pool_kernel_special_scores(values, rule, tau, topk):
    """Ties, infinities and NaN come out as they do from the passes over the matrix (same copies as above)."""
    heads, grid, block = 2, (4, 13, 11), (1, 13, 11)
    small = _shape(heads, grid, block)
    S, Nb = small.S, small.n_blocks
    copies, large = _copies(small)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn((heads, S, Nb), generator=g, device="cuda")
    if values == "constant":
        x.fill_(1.25)
    elif values == "zeros":
        x.zero_()
        x[:, ::3] = -0.0
    elif values == "two":
        x = torch.where(x > 0, 2.0, -1.0)
    elif values == "infinite":
        x[:, ::50] = -float("inf")
        x[0, 7, 1] = float("inf")
    elif values == "nan":
        x[0, 5] = float("nan")
        x[1, 9, 2] = -float("nan")
    score_range = None
    if values == "nan":          # (as the scores kernel leaves it: of the numbers)
        score_range = torch.stack([x.nan_to_num(0.0).amin((1, 2)), x.nan_to_num(0.0).amax((1, 2))], 1).contiguous()
    a = _run(small, x, rule, tau, topk, score_range)
    b = _run(large, _repeat(x, copies), rule, tau, topk, score_range, capacity=int(heads * large.S * Nb))
    ma, mb = _mask(small, a), _mask(large, b).reshape(heads, copies, S, Nb)
    _check_lists(small, a, ma)
    # a NaN takes the mass of the lowest bin of its CTA (there) or thread (here) with it: a few pairs of 600
    assert (ma != mb[:, 0]).sum() <= (8 if values == "nan" else 0) and (mb[:, 0] == mb[:, -1]).all()
    if values == "nan":
        assert np.array_equal(ma[0, 5], mb[0, 0, 5]) and ma[1, 9, 2] == mb[1, 0, 9, 2]


# heads, grid, block, whether the heads go to one cluster each (with fill: two launches): heads of a wave and of several, more than the
# 32 heads before it that a warp adds up at a time; two waves of clusters of eight and of four, of short slices and of long ones
ROUTES = [(33, (4, 8, 8), (1, 8, 8), True), (34, (4, 8, 8), (1, 8, 8), True), (70, (3, 43, 8), (3, 43, 1), True), (149, (4, 8, 8), (1, 8, 8), True),
          (740, (4, 8, 8), (1, 8, 8), True), (741, (4, 8, 8), (1, 8, 8), False),
          (15, (16, 28, 30), (1, 28, 30), True), (16, (16, 28, 30), (1, 28, 30), False), (18, (16, 16, 32), (1, 16, 32), True),
          (33, (16, 19, 30), (1, 19, 30), True), (34, (16, 19, 30), (1, 19, 30), False), (37, (16, 14, 30), (1, 14, 30), True)]


@pytest.mark.parametrize("heads,grid,block,small", ROUTES)
@pytest.mark.parametrize("rule,topk", [(vb.SELECT_THRESHOLD_GLOBAL, 0), (vb.SELECT_TOPK_GLOBAL, 2), (vb.SELECT_TOPK_LOCAL, 2)])
def test_many_heads(heads, grid, block, small, rule, topk):
    """The lists of many heads, on both sides of the rule that gives them to a cluster each; each head's pairs are those that it has
    by itself."""
    shape, one = _shape(heads, grid, block), _shape(1, grid, block)
    S, Nb = shape.S, shape.n_blocks
    g = torch.Generator(device="cuda").manual_seed(heads)
    x = 3.0 * torch.randn((heads, S, Nb), generator=g, device="cuda")
    score_range = torch.stack([x.amin((1, 2)), x.amax((1, 2))], 1).contiguous()
    before = vb.kernel_launches()
    out = _run(shape, x, rule, 0.25, topk, score_range)
    if rule != vb.SELECT_TOPK_LOCAL:
        assert (vb.kernel_launches() - before == 2) == small
    m = _mask(shape, out)
    _check_lists(shape, out, m)
    assert int(out["status"]) == 0
    for h in {0, heads // 3, heads - 2, heads - 1}:
        alone = _run(one, x[h:h + 1].contiguous(), rule, 0.25, topk, score_range[h:h + 1].contiguous())
        # (the cutoff of a mass may fall a pair further: sums of fp32 weights in another order)
        assert (_mask(one, alone)[0] != m[h]).sum() <= (1 if rule == vb.SELECT_THRESHOLD_GLOBAL else 0)


@pytest.mark.parametrize("rule,topk", [(vb.SELECT_TOPK_LOCAL, 3), (vb.SELECT_THRESHOLD_LOCAL, 0),
                                       (vb.SELECT_THRESHOLD_GLOBAL | vb.SELECT_KEEP_OWN_BLOCK, 0)])
@pytest.mark.parametrize("grid,block", SHAPES[1:])
def test_lists_of_small_pools_follow_the_mask(grid, block, rule, topk):
    shape = _shape(3, grid, block)
    x = torch.randn((3, shape.S, shape.n_blocks), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    out = _run(shape, x, rule, 0.3, topk)
    m = _mask(shape, out)
    _check_lists(shape, out, m)
    if rule == vb.SELECT_TOPK_LOCAL:
        want = torch.zeros_like(x, dtype=torch.bool).scatter_(2, x.topk(min(topk, shape.n_blocks), 2).indices, True)
        assert np.array_equal(m, want.cpu().numpy())
        assert torch.equal(out["cutoff"], torch.where(want, x, torch.inf).amin((1, 2)))
    if rule & vb.SELECT_KEEP_OWN_BLOCK:
        own = np.arange(shape.S) // (shape.S // shape.n_blocks)
        assert m[:, np.arange(shape.S), own].all()


def test_too_small_a_capacity_is_reported():
    shape = _shape(2, (4, 8, 8), (1, 8, 8))
    x = torch.randn((2, shape.S, shape.n_blocks), device="cuda")
    out = _run(shape, x, vb.SELECT_TOPK_LOCAL, topk=2, capacity=700)
    assert int(out["status"]) == vb.ERR_CAPACITY
    out = _run(shape, x, vb.SELECT_TOPK_LOCAL, topk=2, capacity=1024)
    assert int(out["status"]) == 0
