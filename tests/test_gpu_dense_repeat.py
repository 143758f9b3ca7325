"""The dense backward adds the parts of dQ key tile after key tile: two runs agree bit for bit, whatever order the CTAs come
in, and the sum is right at the edges of tiles and units, with one head and with more heads than are taken in turn, with one to
four accumulators."""
import pytest
import torch

from paper_2506_23858_b200 import binding as vb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B, heads, S", [(1, 1, 1), (1, 2, 127), (1, 1, 129), (2, 3, 640), (1, 17, 300), (3, 50, 257), (1, 1, 20000),
                                         (1, 12, 5000), (1, 20, 13440)])
def test_dense_gradients_repeat(B, heads, S):
    shape = vb.make_shape(B, heads, 128, (S, 1, 1), (S, 1, 1), "bf16")
    torch.manual_seed(S)
    q, k, v, do = (torch.randn(B, heads, S, 128, device="cuda").to(torch.bfloat16) for _ in range(4))
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(vb.workspace_bytes(shape, vb.STAGE_FULL_BWD), dtype=torch.uint8, device="cuda")
    runs = []
    for fill in (0, 255, 63):                       # what an earlier call left in the workspace does not matter
        ws.fill_(fill)
        o, dq, dk, dv = (torch.full_like(q, 7.0) for _ in range(4))
        lse = torch.empty(B * heads * S, device="cuda")
        vb.vmoba_full_attn(shape, q, k, v, o, lse, do, dq, dk, dv, st, ws)
        runs.append((o, dq, dk, dv))
    assert int(st.item()) == 0
    for other in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(runs[0], other))
    # every gradient of the first and the last head, in fp32 (rounding of P, dS and the results to bf16: 1e-2 in the 2-norm)
    for b, h in {(0, 0), (B - 1, heads - 1)}:
        qf, kf, vf, dof = (x[b, h].float() for x in (q, k, v, do))
        dqs, dkr, dvr = [], torch.zeros_like(kf), torch.zeros_like(vf)
        for i in range(0, S, 2048):
            p = torch.softmax(qf[i:i + 2048] @ kf.T * 128 ** -0.5, dim=1)
            dvr += p.T @ dof[i:i + 2048]
            ds = p * (dof[i:i + 2048] @ vf.T - (p @ vf * dof[i:i + 2048]).sum(1, keepdim=True)) * 128 ** -0.5
            dqs.append(ds @ kf)
            dkr += ds.T @ qf[i:i + 2048]
        for got, ref in ((runs[0][1], torch.cat(dqs)), (runs[0][2], dkr), (runs[0][3], dvr)):
            err = float((got[b, h].float() - ref).norm())
            assert err <= 1e-2 * float(ref.norm()) + 1e-3 * S ** 0.5
