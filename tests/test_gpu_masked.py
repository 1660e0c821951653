"""What a row sees must reach it, and what it does not see must not: NaN, Inf and huge values in q, k and v through every
kernel of the forward and of the multi-token / paged decode.  A row that sees a NaN is NaN; a row that does not is the
row computed without it."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from launched import launched
from oracle import cowa_oracle as orc
from test_gpu_fwd_forms import check_form
from test_gpu_parity import TOL_LSE, check

pytestmark = pytest.mark.gpu
DEV = "cuda"
NAN, INF = float("nan"), float("inf")


def _sees(w, rows, off, keys):
    """[rows, keys] of bool: which of the keys a row of the head with tuple w = (sink, near, gap, len) sees."""
    s, n, g, l = w
    d = (np.asarray(rows)[:, None] + off) - np.asarray(keys)[None, :]
    k = np.asarray(keys)[None, :]
    return (d >= 0) & ((d < n) | (k < s) | ((d >= n + g) & (d < n + g + l)))


# one shape per form of the forward kernels: (B, Nq, Nk, Hq, Hkv, D, sink, local), and the form as test_gpu_fwd_forms names it
FORMS = [
    ((1, 130, 6000, 4, 2, 128, 64, 700), 8),     # an item shared by a cluster of eight blocks
    ((1, 200, 9000, 4, 2, 64, 64, 700), 8),      # the same at D = 64
    ((2, 1100, 4000, 32, 8, 128, 64, 1500), "pair"),  # two heads per block, items taken over
    ((1, 300, 700, 4, 2, 128, 16, 100), 8),      # short lists: some blocks of a cluster have one step, some none
    ((2, 700, 1400, 4, 4, 64, 64, 300), 2),
    ((2, 300, 1300, 5, 5, 128, 64, 300), 4),
    ((2, 600, 2500, 10, 5, 128, 100, 900), "pair, shared item"),
    ((2, 700, 1400, 8, 8, 128, 64, 300), "plain"),
    ((2, 900, 1000, 10, 5, 64, 16, 130), "plain"),
    ((3, 520, 1100, 24, 8, 64, 64, 100), "one buffer"),
    ((2, 700, 1400, 8, 8, 64, 64, 300), "streams"),
]
FORWARD = [shape for shape, _ in FORMS]


@pytest.mark.parametrize("shape,form", FORMS)
def test_the_shapes_below_reach_every_form(shape, form):
    B, Nq, Nk, Hq, Hkv, D, sink, local = shape
    q, k, v = (x.to(DEV) for x in _forward_inputs(B, Nq, Nk, Hq, Hkv, D))
    o, lse = torch.empty_like(q), torch.empty((B, Hq, Nq), device=DEV)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=cowa_inputs.softmax_scale(D))
    check_form(launched(lambda: cowa.cowa_prefill(q, k, v, o, lse, params))[0], D, False, form, -(-Nq // 128) * B * Hq)


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


# ------------------------------------------------------------------ decode of several tokens, contiguous and paged

def _decode(q, kc, vc, lens, params, page=None, hide=None):
    """o, lse of the call; with `page`, the cache goes through a pool of pages, and hide(i) says that page i of a sequence
    is handed out to another request (a page of NaN)."""
    B, Nq, Hq, D = q.shape
    Hkv, Tmax = kc.shape[1], kc.shape[2]
    o = torch.full_like(q, 7.0).to(DEV)
    lse = torch.full((B, Nq, Hq), 7.0, dtype=torch.float32, device=DEV)
    lens_d = torch.tensor(lens, dtype=torch.int32, device=DEV)
    if page is None:
        nbytes = cowa.cowa_decode_multi_workspace_bytes(B, Nq, Tmax, Hq, Hkv, D, params)
        ws = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device=DEV)
        cowa.cowa_decode_multi(q.to(DEV), kc.to(DEV), vc.to(DEV), lens_d, o, lse, params, ws)
    else:
        assert Tmax % page == 0
        npg = Tmax // page
        other = B * npg  # the other request's page
        table = torch.arange(B * npg, dtype=torch.int32).reshape(B, npg)
        kp = torch.full((B * npg + 1, Hkv, page, D), NAN, dtype=torch.bfloat16)
        vp = torch.full_like(kp, NAN)
        for b in range(B):
            for i in range(npg):
                if hide is not None and hide(b, i):
                    table[b, i] = other
                else:
                    kp[b * npg + i], vp[b * npg + i] = kc[b, :, i * page:(i + 1) * page], vc[b, :, i * page:(i + 1) * page]
        nbytes = cowa.cowa_decode_multi_workspace_bytes(B, Nq, Tmax, Hq, Hkv, D, params)
        ws = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device=DEV)
        cowa.cowa_decode_paged(q.to(DEV), kp.to(DEV), vp.to(DEV), table.to(DEV), lens_d, o, lse, params, ws)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    return o.float().cpu(), lse.cpu()


def _decode_inputs(B, Nq, Tmax, Hq, Hkv, D):
    q = cowa_inputs.make_train_inputs(103, B, Nq, Hq, Hkv, D)[0].permute(0, 2, 1, 3).contiguous()
    _, kc, vc, _ = cowa_inputs.make_decode_inputs(104, B, Tmax, Hq, Hkv, D, Tmax, Tmax)
    return q, kc, vc


DECODE = [  # B, Nq, Tmax, Hq, Hkv, D, sink, local, lens, global heads, offset
    (2, 3, 4096, 16, 2, 128, 20, 100, [4001, 2222], 16, 5),  # eight heads per group
    (1, 5, 3072, 8, 2, 128, 7, 70, [3000], 2, 0),            # four
    (2, 8, 2048, 4, 4, 64, 4, 33, [2048, 130], 8, 4),        # one head, D = 64
    (1, 20, 4096, 8, 1, 128, 100, 300, [3777], 8, 6),        # two row tiles
    (6, 2, 8192, 16, 8, 64, 16, 5000, [8192, 8000, 7777, 6500, 8100, 7001], 8, 0),  # many steps between boundary tiles
]


@pytest.mark.parametrize("case", DECODE)
@pytest.mark.parametrize("bad", [NAN, INF])
@pytest.mark.parametrize("page", [None, 16, 64])
def test_decode_keys_that_no_token_sees(case, bad, page):
    """Rows that no token of the call sees hold non-finite values, and pages that no head sees belong to somebody else."""
    B, Nq, Tmax, Hq, Hkv, D, sink, local, lens, hg, off = case
    q, kc, vc = _decode_inputs(B, Nq, Tmax, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale, hkv_global=hg, hkv_offset=off)
    kb, vb, used = kc.clone(), vc.clone(), {}
    for b in range(B):
        ws = orc.default_windows(lens[b], hg, sink, local)[off:off + Hkv]
        for h in range(Hkv):
            seen = _sees(ws[h], np.arange(Nq), lens[b] - Nq, np.arange(Tmax)).any(0)
            assert not seen[:lens[b]].all()
            kb[b, h, ~seen], vb[b, h, ~seen] = bad, bad
            used[b] = used.get(b, False) | seen
    o, lse = _decode(q, kb, vb, lens, params, page, lambda b, i: not used[b][i * page:(i + 1) * page].any())
    f = cowa_inputs.to_f64
    for b in range(B):
        n = lens[b]
        ws = orc.default_windows(n, hg, sink, local)[off:off + Hkv]
        o_ref, lse_ref = orc.forward(f(q[b].permute(1, 0, 2)), f(kc[b, :, :n]), f(vc[b, :, :n]), ws, scale)
        check(f"lse[b={b}]", lse[b].permute(1, 0).numpy(), lse_ref, TOL_LSE, TOL_LSE)
        check(f"o[b={b}]", o[b].permute(1, 0, 2).numpy(), o_ref)


@pytest.mark.parametrize("case", DECODE)
@pytest.mark.parametrize("where", ["q", "k", "v"])
@pytest.mark.parametrize("page", [None, 16])
def test_decode_nan_reaches_the_tokens_that_see_it_and_no_other(case, where, page):
    B, Nq, Tmax, Hq, Hkv, D, sink, local, lens, hg, off = case
    q, kc, vc = _decode_inputs(B, Nq, Tmax, Hq, Hkv, D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=cowa_inputs.softmax_scale(D), hkv_global=hg, hkv_offset=off)
    clean_o, clean_lse = _decode(q, kc, vc, lens, params, page)
    t = Nq // 2
    # the key of token t, and one at the far edge of the near window: the later tokens do not see it any more
    for key in (lens[0] - Nq + t, lens[0] - Nq + t - local + 1):
        qb, kb, vb = q.clone(), kc.clone(), vc.clone()
        if where == "q":
            qb[0, t] = NAN
        else:
            (kb if where == "k" else vb)[0, :, key] = NAN
        o, lse = _decode(qb, kb, vb, lens, params, page)
        for h in range(Hq):
            w = orc.default_windows(lens[0], hg, sink, local)[off + h * Hkv // Hq]
            hit = np.arange(Nq) == t if where == "q" else _sees(w, np.arange(Nq), lens[0] - Nq, [key])[:, 0]
            assert hit[t]
            assert torch.isnan(o[0, hit, h]).all(), f"head {h}: a NaN in {where} came out as a number"
            # the masked weights are exactly zero, so the other tokens differ by the order of their sums at most
            assert torch.isfinite(o[0, ~hit, h]).all()
            assert torch.allclose(o[0, ~hit, h], clean_o[0, ~hit, h], rtol=2.0 ** -7, atol=2.0 ** -8)
            if where != "v":
                assert torch.isnan(lse[0, hit, h]).all()
            assert torch.equal(lse[0, ~hit, h], clean_lse[0, ~hit, h])
        for b in range(1, B):
            assert torch.equal(o[b], clean_o[b]) and torch.equal(lse[b], clean_lse[b])
