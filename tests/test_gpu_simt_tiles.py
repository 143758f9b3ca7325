"""The CUDA-core attention kernels (fp32, and bf16 with head_dim 64) at the edges of their 64 x 64 tiles: key blocks and lists of
one row, of a tile, of one more or fewer, queries without a block, forward and both gradients, sparse and dense.  Against the
same arithmetic in 64 bits: sums of up to 300 fp32 terms are off by 300 * 2^-24 of their largest partial sum at most, 2e-5
relative; bf16 results by their rounding on top, 2^-8 relative."""
import numpy as np
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer, lists_from_mask

pytestmark = pytest.mark.gpu


def _reference(q, k, v, do, mask, scale):
    """q, k, v, do [BH, S, d] in 64 bits; mask [BH, S, S] of the keys a query sees.  o, lse, dq, dk, dv."""
    s = (q @ k.transpose(1, 2)) * scale
    s = s.masked_fill(~mask, -float("inf"))
    lse = torch.logsumexp(s, -1)
    p = torch.exp(s - torch.where(lse.isinf(), torch.zeros_like(lse), lse)[..., None]).masked_fill(~mask, 0.0)
    o = p @ v
    ds = p * (do @ v.transpose(1, 2) - (do * o).sum(-1, keepdim=True))
    return o, lse, ds @ k * scale, ds.transpose(1, 2) @ q * scale, p.transpose(1, 2) @ do


def _close(got, want, dtype, what):
    got, want = got.double(), want
    rel = 2e-5 if dtype == "f32" else 1e-2
    assert not got.isnan().any(), what
    assert float((got - want).norm()) <= rel * float(want.norm()) + 1e-12, (what, float((got - want).norm() / want.norm()))
    assert float((got - want).abs().max()) <= 5 * rel * max(1.0, float(want.abs().max())), what


@pytest.mark.parametrize("d,dtype", [(64, "f32"), (128, "f32"), (64, "bf16")])
@pytest.mark.parametrize("sb,nb", [(1, 5), (31, 3), (32, 4), (33, 3), (63, 3), (64, 4), (65, 3), (130, 2)])
def test_tile_edges(sb, nb, d, dtype):
    heads, S = 2, sb * nb
    shape = vb.make_shape(1, heads, d, (nb, sb, 1), (1, sb, 1), dtype)
    g = torch.Generator(device="cuda").manual_seed(sb * 7 + nb)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    q, k, v, do = (torch.randn((1, heads, S, d), generator=g, device="cuda").to(dt) for _ in range(4))
    # lists of 0, 1, 31 .. 65 and all queries, among them queries with no block and with several
    m = np.zeros((heads, S, nb), dtype=bool)
    rng = np.random.default_rng(sb)
    for h in range(heads):
        for j in range(nb):
            n = [S, 0, 1, min(S, 33), min(S, 65), min(S, 64), min(S, 31)][(h * nb + j) % 7]
            m[h, rng.permutation(S)[:n], j] = True
    m[0, S // 2] = False
    kb_ptr, q_idx, q_ptr, q_pairs, n = lists_from_mask(m)
    L = VmobaLayer(shape, q_idx.numel(), with_backward=True)
    L.kb_ptr, L.q_idx, L.q_ptr, L.q_pairs = kb_ptr, q_idx, q_ptr, q_pairs
    L.q_bm, L.k_bm, L.v_bm, L.do_bm = q, k, v, do
    for x in (L.o_bm, L.dq_bm, L.dk_bm, L.dv_bm):
        x.fill_(float("nan"))
    L.attn_fwd()
    L.attn_bwd()
    torch.cuda.synchronize()
    assert int(L.dev_status.item()) == 0
    mask = torch.from_numpy(np.repeat(m, sb, axis=2)).cuda()
    f = lambda x: x[0].double()
    o, lse, dq, dk, dv = _reference(f(q), f(k), f(v), f(do), mask, d ** -0.5)
    _close(L.o_bm[0], o, dtype, "o")
    got_lse = L.lse.reshape(heads, S).double()
    assert torch.equal(got_lse.isinf(), lse.isinf()) and float((got_lse - lse)[~lse.isinf()].abs().max()) <= 2e-5
    for name, got, want in (("dq", L.dq_bm, dq), ("dk", L.dk_bm, dk), ("dv", L.dv_bm, dv)):
        _close(got[0], want, dtype, name)


@pytest.mark.parametrize("d,dtype", [(64, "f32"), (128, "f32"), (64, "bf16")])
@pytest.mark.parametrize("S", [1, 33, 64, 65, 200])
def test_dense_tile_edges(S, d, dtype):
    heads = 2
    shape = vb.make_shape(1, heads, d, (1, S, 1), (1, S, 1), dtype)
    g = torch.Generator(device="cuda").manual_seed(S)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    q, k, v, do = (torch.randn((1, heads, S, d), generator=g, device="cuda").to(dt) for _ in range(4))
    o, dq, dk, dv = (torch.full_like(q, float("nan")) for _ in range(4))
    lse, status = torch.empty(heads * S, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(vb.workspace_bytes(shape, vb.STAGE_FULL_BWD), dtype=torch.uint8, device="cuda")
    vb.vmoba_full_attn(shape, q, k, v, o, lse, do, dq, dk, dv, status, ws)
    torch.cuda.synchronize()
    f = lambda x: x[0].double()
    want = _reference(f(q), f(k), f(v), f(do), torch.ones((heads, S, S), dtype=torch.bool, device="cuda"), d ** -0.5)
    _close(o[0], want[0], dtype, "o")
    assert float((lse.reshape(heads, S).double() - want[1]).abs().max()) <= 2e-5
    for name, got, w in (("dq", dq, want[2]), ("dk", dk, want[3]), ("dv", dv, want[4])):
        if S > 1 or name == "dv":            # (one key: the weights are 1 and dq, dk are rounding alone)
            _close(got[0], w, dtype, name)
