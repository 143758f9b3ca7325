"""The scratch of a selection is a function of the shape alone: the same number without a GPU, on this one and on another, whichever
route the call takes there."""
import pytest

from paper_2506_23858_b200 import binding as vb

# (B, heads, head_dim, grid, block, type), bytes of STAGE_SELECT, of STAGE_SELECT_ROWNORM: pools of one CTA to eight, and beyond them
SIZES = [
    ((1, 1, 64, (4, 8, 8), (1, 8, 8), "f32"), 58880, 62976),
    ((1, 2, 64, (4, 8, 8), (1, 8, 8), "f32"), 116480, 124672),
    ((1, 12, 128, (6, 12, 26), (3, 6, 13), "bf16"), 716544, 1435392),
    ((1, 12, 128, (21, 20, 32), (21, 5, 8), "bf16"), 1171712, 11493632),
    ((2, 12, 128, (21, 30, 52), (3, 6, 13), "bf16"), 29393920, 469688320),
    ((1, 1, 64, (7, 1024, 1), (7, 1, 1), "f32"), 2110208, 31470336),
    ((1, 40, 128, (21, 45, 80), (1, 45, 80), "bf16"), 18085888, 272101888),
    ((3, 50, 64, (4, 16, 16), (1, 16, 16), "f32"), 8704000, 11161600),
]


def _check():
    for args, select, rownorm in SIZES:
        shape = vb.make_shape(*args)
        assert vb.workspace_bytes(shape, vb.STAGE_SELECT) == select, args
        assert vb.workspace_bytes(shape, vb.STAGE_SELECT_ROWNORM) == rownorm, args


def test_sizes_without_a_gpu():
    _check()


@pytest.mark.gpu
def test_sizes_on_a_gpu():
    _check()


@pytest.mark.gpu
@pytest.mark.parametrize("args,size", [(a, n) for a, n, _ in SIZES if n < 1 << 22])
def test_that_size_is_taken_and_a_smaller_one_refused(args, size):
    import torch
    shape = vb.make_shape(*args)
    BH, S, Nb = shape.B * shape.heads, shape.S, shape.n_blocks
    cap = BH * S * Nb
    x = torch.randn((BH, S, Nb), device="cuda")
    new = lambda n, dt=torch.int32: torch.empty(n, dtype=dt, device="cuda")
    room = torch.full((size + 256,), 0x5a, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    k = new(BH, torch.int64)

    def call(n, rule):
        vb.vmoba_select_rule_apply(shape, x, rule, 0.25, 2, new(BH * S * shape.mask_words), new(BH * Nb + 1), new(cap), new(BH * S + 1),
                                   new(cap), cap, k, new(BH, torch.float32), status, room[:n])

    for rule in (vb.SELECT_THRESHOLD_GLOBAL, vb.SELECT_TOPK_LOCAL):
        call(size, rule)
        torch.cuda.synchronize()
        assert int(status.item()) == 0 and int(k.min()) > 0 and (room[size:] == 0x5a).all()
        with pytest.raises(vb.VmobaError, match="workspace"):
            call(size - 256, rule)
