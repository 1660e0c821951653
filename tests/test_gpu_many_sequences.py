"""GPU tests of packed batches of many sequences: how a work item finds its sequence, in the batch's order and in order of
length, below and above 32 sequences (a second one per lane) and 64 (batch order only), in every form in which the forward
hands out its items, and in the backward with its shared tiles."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from oracle import cowa_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda"
SINK, LOCAL = 130, 300  # more than one sink tile, and sequences shorter than that


def lengths(B, typical):
    """Empty ones, single tokens, equal ones and tile edges among lengths around `typical`, a long one near the end."""
    special = {1: 0, 3: 1, 4: 64, 5: 128, 6: 129, 7: 0}
    n = [special.get(i, typical // 2 + (i * i * 37) % typical) for i in range(B)]
    n[B // 2] = n[B // 2 + 1] = typical
    n[B - 2] = 5 * typical
    return n


def packed(index, H, n, D):
    return cowa_inputs.make_train_inputs(index, 1, sum(n), H, H, D)[0][0]


def run_forward(nq, nk, Hq, Hkv, D, local=LOCAL):
    q, k, v = packed(420, Hq, nq, D), packed(421, Hkv, nk, D), packed(422, Hkv, nk, D)
    params = cowa.make_params(sink=SINK, local=local, softmax_scale=cowa_inputs.softmax_scale(D))
    o = torch.full_like(q, float("nan"), device=DEV)
    lse = torch.full(q.shape[:2], float("nan"), device=DEV)
    cu = [torch.tensor(np.cumsum([0] + n), dtype=torch.int32, device=DEV) for n in (nq, nk)]
    cowa.cowa_prefill_varlen(q.to(DEV), k.to(DEV), v.to(DEV), o, lse, *cu, params)
    torch.cuda.synchronize()
    return q, k, v, o.float().cpu().numpy(), lse.cpu().numpy()


def sequences(nq, nk):
    at_q = at_k = 0
    for a, b in zip(nq, nk):
        yield slice(at_q, at_q + a), slice(at_k, at_k + b)
        at_q, at_k = at_q + a, at_k + b


def close(name, got, want, flat=2e-2, relative=2.0 ** -8):
    """The suite's bounds: max-abs 2e-2 and half a bf16 ulp of the value, for lse 1e-3 and 1e-3 of the value."""
    assert np.isfinite(got).all(), name
    assert (np.abs(got - want) - relative * np.abs(want)).max(initial=0) <= flat, name


@pytest.mark.parametrize("B,typical,prefix,Hq,Hkv,D,local", [
    (32, 40, 50, 4, 2, 64, LOCAL),      # one head a block, by length
    (33, 40, 0, 4, 2, 64, LOCAL),
    (64, 30, 20, 4, 2, 64, LOCAL),
    (65, 30, 20, 4, 2, 64, LOCAL),      # ... in the batch's order
    (100, 20, 0, 4, 2, 64, LOCAL),
    (33, 30, 1100, 32, 2, 128, 2000),   # two heads a block, by length, items taken over
    (64, 20, 1050, 16, 2, 128, 2000),
    (65, 20, 1050, 16, 2, 128, 2000),   # ... in the batch's order
    (34, 110, 0, 32, 2, 128, LOCAL),    # two heads a block, in the batch's order, items in shares and taken over
    (100, 40, 30, 32, 2, 128, LOCAL),
    (8, 400, 0, 32, 2, 128, LOCAL),     # ... by length
])
def test_forward(B, typical, prefix, Hq, Hkv, D, local):
    nq = lengths(B, typical)
    nk = [n + (prefix if i % 3 or prefix > 1000 else 0) for i, n in enumerate(nq)]
    q, k, v, o, lse = run_forward(nq, nk, Hq, Hkv, D, local)
    cowa.cowa_check_device_status()
    f = cowa_inputs.to_f64
    for i, (r, c) in enumerate(sequences(nq, nk)):
        if nq[i]:
            windows = orc.default_windows(nk[i], Hkv, SINK, local)
            want, want_lse = orc.forward(f(q[:, r]), f(k[:, c]), f(v[:, c]), windows, cowa_inputs.softmax_scale(D))
            close(f"o of {i}", o[:, r], want)
            close(f"lse of {i}", lse[:, r], want_lse, 1e-3, 1e-3)


@pytest.mark.parametrize("B,typical", [(34, 110), (100, 40)])
def test_a_malformed_sequence_does_not_hide_the_ones_behind_it(B, typical):
    """More queries than keys in the middle of the batch: reported, and all others as without it."""
    nq, bad = lengths(B, typical), 10
    nk = list(nq)
    nq[bad], nk[bad], nk[0] = 0, 50, nk[0] + 100  # (all together have to have the keys)
    want, want_lse = run_forward(nq, nk, 32, 2, 128)[3:]
    cowa.cowa_check_device_status()
    nq[bad] = 90
    skip = list(sequences(nq, nk))[bad][0]
    others = np.r_[0:skip.start, skip.stop:sum(nq)]
    q = packed(420, 32, [n if i != bad else 0 for i, n in enumerate(nq)], 128)
    whole = torch.zeros(32, sum(nq), 128, dtype=torch.bfloat16)
    whole[:, others] = q
    k, v = packed(421, 2, nk, 128), packed(422, 2, nk, 128)
    params = cowa.make_params(sink=SINK, local=LOCAL, softmax_scale=cowa_inputs.softmax_scale(128))
    o, lse = torch.zeros_like(whole, device=DEV), torch.zeros(whole.shape[:2], device=DEV)
    cu = [torch.tensor(np.cumsum([0] + n), dtype=torch.int32, device=DEV) for n in (nq, nk)]
    cowa.cowa_prefill_varlen(whole.to(DEV), k.to(DEV), v.to(DEV), o, lse, *cu, params)
    torch.cuda.synchronize()
    with pytest.raises(cowa.CowaError) as e:
        cowa.cowa_check_device_status()
    assert e.value.status == -8
    assert np.array_equal(o.float().cpu().numpy()[:, others], want)
    assert np.array_equal(lse.cpu().numpy()[:, others], want_lse)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("B,typical", [(32, 60), (33, 40), (64, 40), (65, 40), (100, 30)])
def test_backward(B, typical, D):
    n, Hq, Hkv = lengths(B, typical), 4, 2
    scale = cowa_inputs.softmax_scale(D)
    q, k, v, d_o = packed(430, Hq, n, D), packed(431, Hkv, n, D), packed(432, Hkv, n, D), packed(433, Hq, n, D)
    dev = [x.to(DEV) for x in (q, k, v)]
    params = cowa.make_params(sink=SINK, local=LOCAL, softmax_scale=scale)
    o, lse = torch.empty_like(dev[0]), torch.empty(q.shape[:2], device=DEV)
    cu = torch.tensor(np.cumsum([0] + n), dtype=torch.int32, device=DEV)
    cowa.cowa_prefill_varlen(*dev, o, lse, cu, cu, params)
    grads = [torch.full_like(x, float("nan")) for x in dev]
    ws = torch.full((cowa.cowa_bwd_varlen_workspace_bytes(B, sum(n), Hq, Hkv, D, params),), 0xFF, dtype=torch.uint8, device=DEV)
    cowa.cowa_bwd_varlen(*dev, o, lse, d_o.to(DEV), *grads, cu, params, ws)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    grads = [x.float().cpu().numpy() for x in grads]
    f = cowa_inputs.to_f64
    for i, (r, _) in enumerate(sequences(n, n)):
        if n[i]:
            want = orc.backward(f(q[:, r]), f(k[:, r]), f(v[:, r]), f(d_o[:, r]), orc.default_windows(n[i], Hkv, SINK, LOCAL), scale)
            for name, got, w in zip(("dq", "dk", "dv"), grads, want):
                close(f"{name} of {i}", got[:, r], w)
