"""Several tensors partitioned by one launch, around the rows a warp takes at a time (8 and 32) and for every row width,
against the index permutation of the oracle; and the dense step of a sampler on tensors that partition as they lie and
on ones that do not."""
import numpy as np
import pytest
import torch

from oracle import vmoba_oracle as orc
from paper_2506_23858_b200 import binding as vb
from paper_2506_23858_b200.layer import SteppedAttention, VmobaLayer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4])
@pytest.mark.parametrize("B, heads, d, dtype, grid, block", [
    (1, 1, 64, "bf16", (1, 1, 1), (1, 1, 1)), (1, 3, 128, "bf16", (1, 3, 3), (1, 3, 1)),
    (2, 2, 64, "f32", (2, 4, 6), (1, 2, 3)), (1, 5, 128, "f32", (3, 5, 7), (3, 1, 7)),
    (2, 12, 128, "bf16", (7, 60, 40), (7, 6, 8))], ids=["one_row", "27_rows", "192_rows", "525_rows", "403k_rows"])
def test_many_tensors_and_tables(n, B, heads, d, dtype, grid, block):
    shape = vb.make_shape(B, heads, d, grid, block, dtype)
    S = shape.S
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    torch.manual_seed(5)
    rasters = [torch.randn(B, S, heads, d, device="cuda").to(dt) for _ in range(n)]
    if n > 1:       # one tensor a slice of a wider one: its own strides
        wide = torch.randn(B, S, heads, 3 * d, device="cuda").to(dt)
        rasters[1] = wide[..., d:2 * d]
    strides = [(x.stride(0), x.stride(1), x.stride(2)) for x in rasters]
    bms = [torch.full((B, heads, S, d), 7.0, dtype=dt, device="cuda") for _ in range(n)]
    perm, inv = (torch.full((S,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    vb.vmoba_partition_many(shape, 0, rasters, bms, strides, perm, inv)
    want, want_inv = orc.partition_perm(*grid, *block)
    assert np.array_equal(perm.cpu().numpy(), want) and np.array_equal(inv.cpu().numpy(), want_inv)
    idx = torch.from_numpy(np.asarray(want)).long().cuda()
    for x, bm in zip(rasters, bms):
        assert torch.equal(bm, x[:, idx].permute(0, 2, 1, 3))
    back = [torch.full_like(x, 3.0).contiguous() for x in rasters]
    vb.vmoba_partition_many(shape, 1, bms, back, [(x.stride(0), x.stride(1), x.stride(2)) for x in back])
    for x, y in zip(rasters, back):
        assert torch.equal(x, y)


def test_number_of_tensors_is_checked():
    shape = vb.make_shape(1, 1, 64, (1, 1, 1), (1, 1, 1), "bf16")
    x = torch.zeros(1, 1, 1, 64, dtype=torch.bfloat16, device="cuda")
    for n in (0, 5):
        with pytest.raises(vb.VmobaError):
            vb.vmoba_partition_many(shape, 0, [x] * n, [x] * n, [(64, 64, 64)] * n)


def test_dense_step_takes_any_strides():
    shape = vb.make_shape(1, 2, 128, (2, 8, 8), (1, 4, 4), "bf16")
    L = VmobaLayer(shape, 4096)
    stepped = SteppedAttention(L, 0.25, 1, 1.0)
    torch.manual_seed(6)
    q, k, v = (torch.randn(1, shape.S, 2, 128, device="cuda").to(torch.bfloat16) for _ in range(3))
    o = torch.empty_like(q)
    assert stepped.forward(0, q, k, v, o) == "dense"
    odd = [x.transpose(2, 3).contiguous().transpose(2, 3) for x in (q, k, v)]       # unit stride along the heads
    o_odd = torch.empty_like(q).transpose(2, 3).contiguous().transpose(2, 3)
    stepped.forward(0, *odd, o_odd)
    L.check_status()
    assert torch.equal(o, o_odd)


@pytest.mark.parametrize("dtype, d", [("bf16", 128), ("f32", 64)])
def test_dense_step_keeps_the_raster_order(dtype, d):
    """Bit for bit full attention over the tokens in the caller's order: a row's weights are rounded against a running
    maximum, so another order of the keys gives other last bits."""
    shape = vb.make_shape(2, 2, d, (6, 12, 26), (3, 6, 13), dtype)
    L = VmobaLayer(shape, 4096)
    torch.manual_seed(8)
    q, k, v = (2.0 * torch.randn(2, shape.S, 2, d, device="cuda").to(L.q_bm.dtype) for _ in range(3))
    o = torch.empty_like(q)
    assert SteppedAttention(L, 0.25, 1, 1.0).forward(0, q, k, v, o) == "dense"
    qh, kh, vh = (x.permute(0, 2, 1, 3).contiguous() for x in (q, k, v))
    ref, lse = torch.empty_like(qh), torch.empty(2 * 2 * shape.S, device="cuda")
    vb.vmoba_full_attn(shape, qh, kh, vh, ref, lse, dev_status=L.dev_status)
    L.check_status()
    assert torch.equal(o, ref.permute(0, 2, 1, 3))


def _placed(x, how):
    """The values of x in a tensor that lies in memory otherwise."""
    if how == "offset":                                     # contiguous, one element off a 16-byte boundary
        y = torch.empty(x.numel() + 1, dtype=x.dtype, device="cuda")[1:].view(x.shape)
    elif how == "batch_stride":                             # one batch whose stride is no multiple of 16 bytes
        y = torch.empty(x.numel(), dtype=x.dtype, device="cuda").as_strided(x.shape, (x.numel() + 3, *x.stride()[1:]))
    else:
        y = torch.empty(x.shape, dtype=how, device="cuda")
    return y.copy_(x)


@pytest.mark.parametrize("how", ["offset", "batch_stride", torch.float32, torch.bfloat16], ids=str)
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_dense_step_takes_any_placement_and_type(dtype, how):
    shape = vb.make_shape(1, 2, 64, (2, 8, 8), (1, 4, 4), dtype)
    L = VmobaLayer(shape, 4096)
    stepped = SteppedAttention(L, 0.25, 1, 1.0)
    torch.manual_seed(6)
    qkv = [torch.randn(1, shape.S, 2, 64, device="cuda").to(torch.bfloat16).to(L.q_bm.dtype) for _ in range(3)]
    o = torch.empty_like(qkv[0])
    stepped.forward(0, *qkv, o)
    o2 = _placed(torch.zeros_like(o), how)
    stepped.forward(0, *[_placed(x, how) for x in qkv], o2)
    L.check_status()
    assert torch.equal(o2, o.to(o2.dtype))


def test_dense_step_takes_expanded_inputs_and_refuses_an_expanded_output():
    shape = vb.make_shape(2, 2, 64, (2, 8, 8), (1, 4, 4), "f32")
    L = VmobaLayer(shape, 4096)
    stepped = SteppedAttention(L, 0.25, 1, 1.0)
    torch.manual_seed(6)
    q, kv = torch.randn(2, shape.S, 2, 64, device="cuda"), torch.randn(1, shape.S, 2, 64, device="cuda")
    o, want = torch.empty_like(q), torch.empty_like(q)
    stepped.forward(0, q, kv.expand_as(q), kv.expand_as(q), o)
    stepped.forward(0, q, kv.expand_as(q).clone(), kv.expand_as(q).clone(), want)
    assert torch.equal(o, want)
    with pytest.raises(RuntimeError):
        stepped.forward(0, q, q, q, torch.empty(1, shape.S, 2, 64, device="cuda").expand_as(q))
