"""NaN scores under the head-wide rules: one without a sign has the place of -0, one with a sign lies below every number, and what
they weigh is left out of the mass; so a few of them change the selection of the other pairs by a few.  The same on every route
(one cluster per head; passes over the matrix), with and without a range from the scores kernel."""
import numpy as np
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from tests.test_gpu_select_pool import _check_lists, _mask, _run, _shape

pytestmark = pytest.mark.gpu

SHAPES = {"one CTA": ((4, 13, 11), (1, 13, 11)), "four CTAs": ((6, 12, 26), (3, 6, 13)), "eight CTAs": ((16, 16, 16), (2, 8, 8)),
          "passes": ((64, 32, 32), (4, 32, 32))}


def _keys(x):
    u = x.view(np.uint32)
    key = np.where(u & 0x80000000, ~u, u | 0x80000000)
    return np.where(key > 0xff800000, np.uint32(0x7fffffff), key)


@pytest.mark.parametrize("route", SHAPES)
@pytest.mark.parametrize("rule,tau,topk", [(vb.SELECT_THRESHOLD_GLOBAL, 0.25, 0), (vb.SELECT_THRESHOLD_GLOBAL, 0.9, 0),
                                           (vb.SELECT_THRESHOLD_GLOBAL, 1.0, 0), (vb.SELECT_TOPK_GLOBAL, 0.0, 2)])
@pytest.mark.parametrize("ranged", [False, True])
@pytest.mark.parametrize("signs", ["none", "minus", "both"])
def test_nan_scores(route, rule, tau, topk, ranged, signs):
    heads = 3
    shape = _shape(heads, *SHAPES[route])
    S, Nb = shape.S, shape.n_blocks
    x = torch.randn((heads, S, Nb), generator=torch.Generator(device="cuda").manual_seed(11), device="cuda")
    x[2] = torch.exp(x[2])                                         # (positive numbers: cutoffs above -0)
    score_range = torch.stack([x.amin((1, 2)), x.amax((1, 2))], 1).contiguous() if ranged else None
    clean = _run(shape, x, rule, tau, topk, score_range)
    nan, neg = np.float32(np.nan), np.uint32(0xffc00000).view(np.float32)
    h = x.cpu().numpy()
    n_nan = 0
    for head in range(heads):
        if signs != "minus":
            h[head, 5] = nan
            n_nan += Nb
        if signs != "none":
            h[head, 9, 1] = h[head, 17, 0] = neg
            n_nan += 2
    y = torch.from_numpy(h).cuda()
    out = _run(shape, y, rule, tau, topk, score_range)
    m = _mask(shape, out)
    _check_lists(shape, out, m)
    assert int(out["status"]) == 0
    cut = out["cutoff"].cpu().numpy()
    # what the cutoff says of every pair, NaN or not
    assert np.array_equal(m, _keys(h) >= _keys(cut)[:, None, None])
    if signs == "none" or ranged:
        # the numbers' selection: that without the NaN, but for the bin that their mass is lost with (the lowest of a CTA) and, for a
        # budget of pairs, for their number
        ok = ~np.isnan(h)
        was, now = (_mask(shape, clean) & ok).sum((1, 2)), (m & ok).sum((1, 2))
        assert (np.abs(was - now) <= max(n_nan, 0.01 * S * Nb)).all(), (was, now)
