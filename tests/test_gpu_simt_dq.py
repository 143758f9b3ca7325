"""dq of the sparse CUDA-core backward (fp32, and bf16 with head_dim 64).  A query's row of it is the sum of one part per selected
block, each part worked out in a fixed order: a query with one or two blocks has the same dq in every call, whatever the order in
which the parts come.  And dq may lie over an input: it is written when everything that is read has been."""
import numpy as np
import pytest
import torch

from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import VmobaLayer, lists_from_mask

pytestmark = pytest.mark.gpu


def _layer(sb, nb, d, dtype, heads=3, seed=0):
    S = sb * nb
    shape = vb.make_shape(1, heads, d, (nb, sb, 1), (1, sb, 1), dtype)
    g = torch.Generator(device="cuda").manual_seed(sb + nb + seed)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    x = [torch.randn((1, heads, S, d), generator=g, device="cuda").to(dt) for _ in range(4)]
    # blocks per query: 0, 1, 2, 1, 2, .. and every ninth query all of them
    m = np.zeros((heads, S, nb), dtype=bool)
    rng = np.random.default_rng(seed)
    for h in range(heads):
        for i in range(S):
            n = nb if i % 9 == 8 else min(nb, i % 3)
            m[h, i, rng.permutation(nb)[:n]] = True
    kb_ptr, q_idx, q_ptr, q_pairs, _ = lists_from_mask(m)
    L = VmobaLayer(shape, q_idx.numel(), with_backward=True)
    L.kb_ptr, L.q_idx, L.q_ptr, L.q_pairs = kb_ptr, q_idx, q_ptr, q_pairs
    L.q_bm, L.k_bm, L.v_bm, L.do_bm = x
    L.attn_fwd()
    return L, torch.from_numpy(m.sum(2)).cuda()


@pytest.mark.parametrize("d,dtype", [(64, "f32"), (128, "f32"), (64, "bf16")])
@pytest.mark.parametrize("sb,nb", [(48, 7), (64, 6), (65, 5), (128, 4), (129, 4), (200, 4), (449, 3), (512, 3), (513, 3), (720, 3)])
def test_queries_of_one_or_two_blocks_repeat(sb, nb, d, dtype):
    L, blocks = _layer(sb, nb, d, dtype)
    L.attn_bwd()
    first = [x.clone() for x in (L.dq_bm, L.dk_bm, L.dv_bm)]
    few = blocks <= 2
    # the sums of many parts differ in their last bits from call to call; they are fp32 sums of at most nb parts
    for _ in range(30):
        for x in (L.dq_bm, L.dk_bm, L.dv_bm):
            x.fill_(float("nan"))
        L.attn_bwd()
        assert torch.equal(L.dk_bm, first[1]) and torch.equal(L.dv_bm, first[2])
        assert torch.equal(L.dq_bm[0][few], first[0][0][few])
        assert torch.allclose(L.dq_bm.float(), first[0].float(), rtol=2.0 ** -7, atol=1e-4)
    assert (first[0][0][blocks == 0] == 0).all()
    L.check_status()


@pytest.mark.parametrize("sb,nb", [(64, 4), (130, 3)])
@pytest.mark.parametrize("shift", [0, 4, 64 * 5, -64 * 5])
@pytest.mark.parametrize("over", ["q_bm", "k_bm", "v_bm", "o_bm", "do_bm", "lse", "kb_ptr", "q_idx"])
def test_dq_may_lie_over_an_input(over, shift, sb, nb):
    d = 64
    L, blocks = _layer(sb, nb, d, "f32", heads=2, seed=5)
    L.attn_bwd()
    want, dk, dv = L.dq_bm.clone(), L.dk_bm.clone(), L.dv_bm.clone()
    src = getattr(L, over)
    n, pad = want.numel(), 1024
    room = torch.zeros(max(n, src.numel()) + 2 * pad, device="cuda")
    at = room[pad:pad + src.numel()].view(src.dtype).view(src.shape)
    at.copy_(src)
    setattr(L, over, at)
    L.dq_bm = room[pad + shift:pad + shift + n].view(want.shape)
    L.attn_bwd()
    L.check_status()
    few = blocks <= 2
    assert torch.equal(L.dk_bm, dk) and torch.equal(L.dv_bm, dv)
    assert torch.equal(L.dq_bm[0][few], want[0][few])
    assert torch.allclose(L.dq_bm, want, rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("d,dtype", [(64, "f32"), (128, "f32"), (64, "bf16")])
def test_long_blocks(d, dtype):
    """Blocks of 57 tiles of keys: sums of 3,600 terms in fp32, against 64 bits."""
    sb, nb, heads = 3600, 2, 2
    L, blocks = _layer(sb, nb, d, dtype, heads=heads, seed=9)
    L.attn_bwd()
    L.check_status()
    m = torch.zeros((heads, sb * nb, nb), dtype=torch.bool, device="cuda")
    kb, qi = L.kb_ptr.tolist(), L.q_idx
    for i in range(heads * nb):
        m[i // nb, qi[kb[i]:kb[i + 1]].long(), i % nb] = True
    for h in range(heads):
        q, k, v, do = (x[0, h].double() for x in (L.q_bm, L.k_bm, L.v_bm, L.do_bm))
        s = (q @ k.T) * d ** -0.5
        s = s.masked_fill(~m[h].repeat_interleave(sb, 1), -float("inf"))
        p = torch.softmax(s, -1).nan_to_num(0.0)
        ds = p * (do @ v.T - (do * (p @ v)).sum(-1, keepdim=True))
        want = ds @ k * d ** -0.5
        err = float((L.dq_bm[0, h].double() - want).norm() / want.norm())
        # 3,600 roundings of 2^-24 would be 2e-4 if all went one way; at random sixty of them, and the bf16 result's own
        assert err <= (1e-5 if dtype == "f32" else 4e-3), err


@pytest.mark.parametrize("sb,nb", [(64, 4), (200, 4), (720, 3)])
def test_a_captured_backward_replays(sb, nb):
    """The three routes of dq in a graph: what it writes is what the call writes."""
    L, blocks = _layer(sb, nb, 64, "f32", seed=2)
    L.attn_bwd()
    torch.cuda.synchronize()
    want = [x.clone() for x in (L.dq_bm, L.dk_bm, L.dv_bm)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        L.attn_bwd()
    for _ in range(3):
        for x in (L.dq_bm, L.dk_bm, L.dv_bm):
            x.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(L.dk_bm, want[1]) and torch.equal(L.dv_bm, want[2])
        assert torch.equal(L.dq_bm[0][blocks <= 2], want[0][0][blocks <= 2])
    L.check_status()
