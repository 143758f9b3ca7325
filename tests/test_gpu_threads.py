"""Calls from several threads of one process: what a kernel may have of shared memory is one setting for all of them, and a
thread's small call must not take it away from another thread's large one."""
import threading

import pytest
import torch

from paper_2506_23858_b200 import binding as vb

pytestmark = pytest.mark.gpu


def _shape(heads, grid, block):
    return vb.make_shape(1, heads, 64, grid, block, "f32")


def _select(shape, rule, topk, heads_of):
    """A selection of the shape's size with everything that it writes; raises where the library reports an error."""
    BH, S, Nb = shape.heads, shape.S, shape.n_blocks
    cap = BH * S * Nb
    x = torch.randn((BH, S, Nb), generator=torch.Generator(device="cuda").manual_seed(heads_of), device="cuda")
    new = lambda n, dt=torch.int32: torch.empty(n, dtype=dt, device="cuda")
    mask = new(BH * S * shape.mask_words)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    keep = (new(BH * Nb + 1), new(cap), new(BH * S + 1), new(cap), new(BH, torch.int64), new(BH, torch.float32), new(1).zero_(),
            new(vb.workspace_bytes(shape, vb.STAGE_SELECT, cap), torch.uint8))
    kb_ptr, q_idx, q_ptr, q_pairs, k, cutoff, status, ws = keep
    torch.cuda.current_stream().synchronize()
    vb.vmoba_select_rule_apply(shape, x, rule, 0.25, topk, mask, kb_ptr, q_idx, q_ptr, q_pairs, cap, k, cutoff, status, ws,
                               stream=stream)
    stream.synchronize()
    assert int(status.item()) == 0
    return k.tolist()


# (grid, block) of the call with the larger and of that with the smaller need, by route: one cluster per head; the passes over the
# matrix (more scores per head than the cluster takes); the per-query rule's mask through either
ROUTES = {
    "pool": (((8, 24, 35), (2, 3, 35)), ((6, 12, 26), (3, 6, 13)), vb.SELECT_THRESHOLD_GLOBAL, 0),
    "passes": (((32, 32, 16), (2, 2, 4)), ((64, 64, 64), (32, 64, 64)), vb.SELECT_THRESHOLD_GLOBAL, 0),
    "top-k": (((32, 32, 16), (2, 2, 4)), ((4, 8, 8), (1, 8, 8)), vb.SELECT_TOPK_LOCAL, 3),
}


@pytest.mark.parametrize("route", ROUTES)
def test_a_small_call_leaves_another_threads_large_calls_alone(route):
    (g1, b1), (g2, b2), rule, topk = ROUTES[route]
    large, small = _shape(2, g1, b1), _shape(2, g2, b2)
    first, second = threading.Event(), threading.Event()
    got, errors = {}, []

    def a():
        try:
            got["before"] = _select(large, rule, topk, 1)
            first.set()
            second.wait(60)
            got["after"] = _select(large, rule, topk, 1)
        except Exception as e:      # noqa: BLE001 (handed to the test's own thread)
            errors.append(("large", e))
            first.set()

    def b():
        try:
            first.wait(60)
            got["small"] = _select(small, rule, topk, 2)
        except Exception as e:      # noqa: BLE001
            errors.append(("small", e))
        second.set()

    threads = [threading.Thread(target=f) for f in (a, b)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not errors, errors
    assert got["before"] == got["after"] and min(got["small"]) > 0


def test_many_threads_at_once():
    shapes = [_shape(2, *ROUTES[r][i]) for r in ROUTES for i in (0, 1)] * 2
    want = [_select(s, vb.SELECT_THRESHOLD_GLOBAL, 0, 3) for s in shapes]
    got, errors = [None] * len(shapes), []

    def work(i):
        try:
            for _ in range(5):
                got[i] = _select(shapes[i], vb.SELECT_THRESHOLD_GLOBAL, 0, 3)
        except Exception as e:      # noqa: BLE001
            errors.append((i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not errors, errors
    for g, w in zip(got, want):      # (a pair at the cutoff may depend on the order of fp32 sums)
        assert all(abs(x - y) <= 1 for x, y in zip(g, w))
