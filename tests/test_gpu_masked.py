"""What a row sees must reach it, and what it does not see must not: NaN, Inf and huge values in q, k and v through every
kernel of the forward.  A row that sees a NaN is NaN; a row that does not is the row computed without it."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from oracle import cowa_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda"
NAN, INF = float("nan"), float("inf")


def _sees(w, rows, off, keys):
    """[rows, keys] of bool: which of the keys a row of the head with tuple w = (sink, near, gap, len) sees."""
    s, n, g, l = w
    d = (np.asarray(rows)[:, None] + off) - np.asarray(keys)[None, :]
    k = np.asarray(keys)[None, :]
    return (d >= 0) & ((d < n) | (k < s) | ((d >= n + g) & (d < n + g + l)))


# one shape per forward kernel: (B, Nq, Nk, Hq, Hkv, D, sink, local)
FORWARD = [
    (1, 130, 6000, 4, 2, 128, 64, 700),     # an item shared by a cluster of eight blocks
    (1, 200, 9000, 4, 2, 64, 64, 700),      # the same at D = 64
    (2, 1100, 4000, 32, 8, 128, 64, 1500),  # two heads per persistent block
    (1, 300, 700, 4, 2, 128, 16, 100),      # one head per block
]


def _forward(q, k, v, sink, local):
    B, Hq, Nq, D = q.shape
    o = torch.full_like(q, 7.0)
    lse = torch.full((B, Hq, Nq), 7.0, dtype=torch.float32, device=DEV)
    cowa.cowa_prefill(q, k, v, o, lse, cowa.make_params(sink=sink, local=local, softmax_scale=cowa_inputs.softmax_scale(D)))
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    return o.float().cpu(), lse.cpu()


def _forward_inputs(B, Nq, Nk, Hq, Hkv, D):
    q = cowa_inputs.make_train_inputs(101, B, Nq, Hq, Hkv, D)[0]
    _, k, v, _ = cowa_inputs.make_train_inputs(102, B, Nk, Hq, Hkv, D)
    return q, k, v


@pytest.mark.parametrize("shape", FORWARD)
@pytest.mark.parametrize("where", ["q", "k", "v"])
def test_forward_nan_reaches_every_row_that_sees_it(shape, where):
    B, Nq, Nk, Hq, Hkv, D, sink, local = shape
    q, k, v = _forward_inputs(B, Nq, Nk, Hq, Hkv, D)
    clean_o, clean_lse = _forward(q.to(DEV), k.to(DEV), v.to(DEV), sink, local)
    rows, key = np.arange(Nq), Nk - Nq // 2  # a key of the chunk itself: some rows see it, the ones before do not
    if where == "q":
        q[0, :, 5] = NAN
    else:
        (k if where == "k" else v)[0, :, key] = NAN
    o, lse = _forward(q.to(DEV), k.to(DEV), v.to(DEV), sink, local)
    ws = orc.default_windows(Nk, Hkv, sink, local)
    for h in range(Hq):
        hit = rows == 5 if where == "q" else _sees(ws[h * Hkv // Hq], rows, Nk - Nq, [key])[:, 0]
        assert hit.any() and not hit.all()
        assert torch.isnan(o[0, h, hit]).all(), f"head {h}: a NaN in {where} came out as a number"
        if where != "v":  # v of a visited tile also meets the rows whose weight for it is zero
            assert torch.isnan(lse[0, h, hit]).all()
            assert torch.equal(o[0, h, ~hit], clean_o[0, h, ~hit]) and torch.equal(lse[0, h, ~hit], clean_lse[0, h, ~hit])
        else:
            assert torch.equal(lse[0, h], clean_lse[0, h])
    for b in range(1, B):
        assert torch.equal(o[b], clean_o[b]) and torch.equal(lse[b], clean_lse[b])


@pytest.mark.parametrize("shape", FORWARD)
def test_forward_inf_value_reaches_every_row_that_sees_it(shape):
    B, Nq, Nk, Hq, Hkv, D, sink, local = shape
    q, k, v = _forward_inputs(B, Nq, Nk, Hq, Hkv, D)
    v[0, :, 3] = INF  # a sink key: every row sees it, and of a shared item one block only
    o, lse = _forward(q.to(DEV), k.to(DEV), v.to(DEV), sink, local)
    assert not torch.isfinite(o[0]).any() and torch.isfinite(lse).all()


@pytest.mark.parametrize("shape", FORWARD)
def test_forward_masked_keys_weigh_exactly_nothing(shape):
    B, Nq, Nk, Hq, Hkv, D, sink, local = shape
    q, k, v = _forward_inputs(B, Nq, Nk, Hq, Hkv, D)
    clean_o, clean_lse = _forward(q.to(DEV), k.to(DEV), v.to(DEV), sink, local)
    first = Nq // 2 - (Nk - Nq + Nq // 2) % 64 + 8  # the rows before it see none of the keys from here on: column 8 of a tile
    assert first > 0 and (Nk - Nq + first) % 64 == 8
    v[:, :, Nk - Nq + first:] = 3e38
    o, lse = _forward(q.to(DEV), k.to(DEV), v.to(DEV), sink, local)
    assert torch.equal(o[:, :, :first], clean_o[:, :, :first]) and torch.equal(lse, clean_lse)
