"""The tensor router's route events over the sizes at which its launches
change: expert chunks (few to many 128-row tiles, 16 to 512 experts),
selection with and without the scatter, row chunks through a small
scratch, misaligned router weights, exact ties, and rows whose top experts
share few lanes of the selecting warp.

Reference: fp64 logits, stable descending sort (equal logits: lower id first).
"""
import numpy as np
import pytest
import torch

from paper_2608_23805_gb300 import api

pytestmark = pytest.mark.gpu


def tolerance(logits, H):
    """The products are exact; each of a logit's 3 H / 16 accumulations drops at
    most one unit in the last place (2^-23) of the running sum.  Four times
    their random sum, at the largest logit; closer pairs may swap."""
    return 4 * 2.0 ** -23 * (3 * H / 16) ** 0.5 * max(1.0, np.abs(logits).max())


def route(x, wr, E, k, H, shared=False):
    """The route event of a forward over a plan with nothing resident (the call
    fails closed after routing)."""
    windows = torch.zeros(64, dtype=torch.uint8, pin_memory=True)
    sw = torch.zeros(3 * 128 * H, dtype=torch.bfloat16, device="cuda") if shared else None
    gw = torch.zeros(1, H, device="cuda") if shared else None
    plan = api.Plan(n_layers=1, n_experts=E, top_k=k, hidden=H, inter=128, n_slots=2, host_windows=windows,
                    has_shared=shared, shared_w=sw, shared_gate_w=gw)
    none = np.full(E, -1, dtype=np.int32)
    _, ev = plan.forward(0, x, wr, none, np.zeros(E, dtype=np.uint64))
    torch.cuda.synchronize()
    got = [t.cpu().numpy() for t in (ev.ids, ev.weights, ev.counts, ev.gap)]
    plan.close()
    return got


def check(x, wr, k, got):
    ids, w, counts, gap = got
    logits = x.double().cpu().numpy() @ wr.double().cpu().numpy().T
    E = logits.shape[1]
    order = np.argsort(-logits, axis=1, kind="stable")
    top = np.take_along_axis(logits, order, 1)
    n = min(k + 1, E)
    d = top[:, :n - 1] - top[:, 1:n] if n > 1 else np.ones((len(top), 1))
    tol = tolerance(logits, x.shape[1])
    clear = ((d == 0) | (d > 2 * tol)).all(axis=1)
    assert clear.mean() >= 0.7  # most rows decide the order
    assert (ids[clear] == order[clear, :k]).all()
    e = np.exp(top[:, :k] - top[:, :1])
    assert np.abs(w - e / e.sum(1, keepdims=True)).max() <= tol
    assert (counts == np.bincount(ids.ravel(), minlength=E)).all()
    if k < E:
        assert np.abs(gap - (top[:, k - 1] - top[:, k])).max() <= 2 * tol
    else:
        assert np.isinf(gap).all()


def inputs(T, E, H, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(T, H, generator=g, device="cuda").to(torch.bfloat16)
    wr = torch.randn(E, H, generator=g, device="cuda") * 0.02
    n = min(4, E // 2)
    wr[E // 2:E // 2 + n] = wr[:n]  # exact ties between experts
    x[T // 2] = 0                   # and over all of them
    return x, wr


@pytest.mark.parametrize("T", [1, 8, 9, 127, 129, 255, 256, 257, 600, 1000, 2049, 4095, 4096, 4097])
def test_lengths(T):
    x, wr = inputs(T, 512, 2048)
    check(x, wr, 10, route(x, wr, 512, 10, 2048, shared=T in (9, 4097)))


@pytest.mark.parametrize("E,k,H", [(48, 10, 1024), (80, 1, 512), (96, 31, 1024), (128, 8, 256), (256, 16, 768),
                                   (384, 6, 256), (512, 1, 256)])
@pytest.mark.parametrize("T", [3, 300, 5000])
def test_shapes(T, E, k, H):
    # (512, 1, 256) at 5,000 rows: the logits' scratch holds fewer rows than the call
    x, wr = inputs(T, E, H, 1)
    check(x, wr, k, route(x, wr, E, k, H))


@pytest.mark.parametrize("E,k,H", [(512, 10, 2048), (128, 8, 256), (48, 4, 1024)])
def test_event_does_not_depend_on_the_call(E, k, H):
    # a row decoded alone, in a small batch and in a prefill: the same bits
    x, wr = inputs(300, E, H, 6)
    whole = route(x, wr, E, k, H)
    for T in (1, 7, 33, 64, 65, 128, 257):
        ids, w, _, gap = route(x[:T], wr, E, k, H)
        assert (ids == whole[0][:T]).all()
        assert (w.view(np.uint32) == whole[1][:T].view(np.uint32)).all()
        assert (gap.view(np.uint32) == whole[3][:T].view(np.uint32)).all()


@pytest.mark.parametrize("T", [5, 700])
@pytest.mark.parametrize("k", [10, 31])
def test_top_experts_in_few_lanes(T, k):
    # experts 128 i + 0 .. 7 lead on every row: two lanes hold the top 32
    x, wr = inputs(T, 512, 512, 2)
    if k == 31:
        wr = wr[:128].clone()
    x = x.abs()
    lead = torch.arange(wr.shape[0], device="cuda") % 128 < 8
    wr[lead] = wr[lead].abs() + 0.05
    check(x, wr, k, route(x, wr, wr.shape[0], k, 512))


@pytest.mark.parametrize("T", [5, 700])
def test_misaligned_router_weights(T):
    x, wr = inputs(T, 512, 512, 3)
    buf = torch.empty(wr.numel() + 1, device="cuda")
    off = buf[1:].view(512, 512)
    off.copy_(wr)
    assert off.data_ptr() % 16 == 4
    check(x, off, 10, route(x, off, 512, 10, 512))


@pytest.mark.parametrize("E,k,H", [(16, 2, 256), (5, 5, 512), (20, 3, 256), (32, 10, 1024)])
@pytest.mark.parametrize("T", [1, 32, 33, 200, 256, 257])
def test_small_layers(T, E, k, H):
    # up to 256 rows the selecting launch scatters too (a cluster of 32-row blocks)
    x, wr = inputs(T, E, H, 4)
    check(x, wr, k, route(x, wr, E, k, H, shared=T == 33))


@pytest.mark.parametrize("E,H", [(16, 256), (512, 512)])
@pytest.mark.parametrize("T", [40, 700])
def test_nan_rows_name_experts(T, E, H):
    # a row without an order still names k different experts, and the others
    # are not touched
    x, wr = inputs(T, E, H, 5)
    x[3] = float("nan")
    ids, w, counts, _ = route(x, wr, E, 2, H)
    assert ids.min() >= 0 and ids.max() < E and (ids[:, 0] != ids[:, 1]).all()
    assert (counts == np.bincount(ids.ravel(), minlength=E)).all()
    assert np.isfinite(np.delete(w, 3, 0)).all()
