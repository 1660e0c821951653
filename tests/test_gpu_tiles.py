"""Sizes at which the two-head forward kernel, its cluster-shared form and the tile decode kernel can go wrong: edges of
128-row tiles, odd numbers of 64-key tiles, the cluster sizes, several row tiles per KV head, many pieces per unit.
Tolerances are those of the parity tests."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from launched import launched
from oracle import cowa_oracle as orc
from test_gpu_parity import TOL_LSE, check, multi_case, _packed_inputs, _run_varlen

pytestmark = pytest.mark.gpu
DEV = "cuda"


# What a call may ask for besides the default rule: (parameters, the windows of an Nk-token sequence)
MODES = {
    "default": lambda Hkv, sink, local: (dict(sink=sink, local=local), lambda Nk: orc.default_windows(Nk, Hkv, sink, local)),
    "full": lambda Hkv, sink, local: (dict(sink=sink, local=local, full_attn=True), lambda Nk: [(0, Nk, 0, 0)] * Hkv),
    # the local heads are some of three times as many
    "rank": lambda Hkv, sink, local: (dict(sink=sink, local=local, hkv_global=3 * Hkv, hkv_offset=Hkv + 1),
                                      lambda Nk: orc.default_windows(Nk, 3 * Hkv, sink, local)[Hkv + 1:2 * Hkv + 1]),
    # tuples of their own for every head: gap or none, wide sink or none, no long window at all
    "tuples": lambda Hkv, sink, local: (lambda ws: (dict(windows=ws), lambda Nk: ws))(
        [[(0, 1500, 300, 1100), (200, 70, 0, 2000), (130, 1700, 0, 0), (1, 1, 65, 1800)][h % 4] for h in range(Hkv)]),
}


def _prefill(B, Nq, Nk, Hq, Hkv, D, sink, local, token_major=False, rows=None, mode="default"):
    q, _, _, _ = cowa_inputs.make_train_inputs(91, B, Nq, Hq, Hkv, D)
    _, k, v, _ = cowa_inputs.make_train_inputs(92, B, Nk, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    kw, windows = MODES[mode](Hkv, sink, local)
    params = cowa.make_params(softmax_scale=scale, **kw)
    put = lambda x: x.to(DEV)  # noqa: E731
    if token_major:
        put = lambda x: x.transpose(1, 2).contiguous().to(DEV).transpose(1, 2)  # noqa: E731
    qd = put(q)
    o = torch.full_like(qd, float("nan"))
    lse = torch.full((B, Hq, Nq), float("nan"), dtype=torch.float32, device=DEV)
    kd, vd = put(k), put(v)
    kernel = launched(lambda: cowa.cowa_prefill(qd, kd, vd, o, lse, params))[0]
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    assert torch.isfinite(o).all() and torch.isfinite(lse).all()
    ws = windows(Nk)
    f = cowa_inputs.to_f64
    rows = np.arange(Nq) if rows is None else np.asarray(rows)
    for b in range(B):
        for h in range(0, Hq, max(1, Hq // 4)):
            o_ref, lse_ref = orc.forward_rows(f(q[b]), f(k[b]), f(v[b]), ws, scale, h, rows)
            check(f"lse[{b},{h}]", lse[b, h].cpu().numpy()[rows], lse_ref, TOL_LSE, TOL_LSE)
            check(f"o[{b},{h}]", o[b, h].float().cpu().numpy()[rows], o_ref)
    return kernel


@pytest.mark.parametrize("B,Nq,Nk,Hq,Hkv,D,sink,local", [
    (1, 130, 6000, 4, 2, 128, 64, 700),    # clusters of 8, last tile of two rows
    (1, 1, 9000, 2, 1, 128, 0, 64),        # one query, one item
    (2, 128, 3000, 8, 2, 128, 130, 333),   # clusters of 8, whole tiles
    (2, 300, 2999, 32, 8, 128, 5, 1500),   # more than half an item per SM: one block per item
    (1, 257, 7000, 8, 4, 64, 64, 500),     # the shared form at D = 64
])
def test_few_items(B, Nq, Nk, Hq, Hkv, D, sink, local):
    _prefill(B, Nq, Nk, Hq, Hkv, D, sink, local)


@pytest.mark.parametrize("mode", ["full", "rank", "tuples"])
@pytest.mark.parametrize("B,Nq,Nk,Hq,Hkv,D", [
    (1, 130, 6000, 8, 4, 128),    # an item shared by a cluster
    (1, 200, 5000, 8, 4, 64),     # the same at D = 64
    (2, 1100, 3000, 32, 4, 128),  # persistent blocks
])
def test_window_modes(B, Nq, Nk, Hq, Hkv, D, mode):
    n = Nq - 1
    _prefill(B, Nq, Nk, Hq, Hkv, D, 64, 1500, mode=mode, rows=[0, 1, 63, 127, 128, 129, n - 1, n])


def test_few_items_token_major():
    _prefill(2, 200, 4000, 8, 2, 128, 64, 500, token_major=True)


@pytest.mark.parametrize("Nq,Nk,sink,local", [
    (4000, 4000, 64, 64),      # short lists, odd and even numbers of key tiles, several items per block
    (3969, 4100, 0, 1),        # near window of one key, last tile of one row
    (2560, 2560, 200, 2000),   # every tile of the longest list visited
])
def test_many_items(Nq, Nk, sink, local):
    n = Nq - 1
    _prefill(2, Nq, Nk, 32, 8, 128, sink, local, rows=[0, 1, 63, 64, 127, 128, 129, n // 2, n - 128, n - 1, n])


@pytest.mark.parametrize("seqs,Hq,Hkv,D", [
    ([(300, 5000), (1, 700), (129, 9000)], 4, 2, 128),                       # clusters share the items of a packed batch
    ([(1900, 1900), (64, 64), (2000, 2500), (1, 3000), (127, 127)], 32, 8, 128),  # one block per item
    ([(200, 9000), (1, 5000), (130, 7000)], 4, 2, 64),                       # clusters at D = 64
])
@pytest.mark.parametrize("bad", [None, float("nan"), float("inf")])
def test_packed(seqs, Hq, Hkv, D, bad):
    """Packed batches against the oracle; with `bad`, one sequence is filled with it and the others must not notice."""
    q, k, v, cu_q, cu_k = _packed_inputs(93, seqs, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=20, local=900, softmax_scale=scale)
    if bad is not None:
        k[:, cu_k[1]:cu_k[2]] = bad
        v[:, cu_k[1]:cu_k[2]] = bad
    o, lse = _run_varlen(q, k, v, cu_q, cu_k, params)
    cowa.cowa_check_device_status()
    f = cowa_inputs.to_f64
    for b, (nq, nk) in enumerate(seqs):
        if bad is not None and b == 1:
            continue
        qs, ks = slice(cu_q[b], cu_q[b + 1]), slice(cu_k[b], cu_k[b + 1])
        ws = orc.default_windows(nk, Hkv, 20, 900)
        for h in (0, Hq - 1):
            o_ref, lse_ref = orc.forward_rows(f(q[:, qs]), f(k[:, ks]), f(v[:, ks]), ws, scale, h, np.arange(nq))
            check(f"lse[{b},{h}]", lse[h, qs].cpu().numpy(), lse_ref, TOL_LSE, TOL_LSE)
            check(f"o[{b},{h}]", o[h, qs].float().cpu().numpy(), o_ref)


@pytest.mark.parametrize("mode", ["full", "rank", "tuples"])
@pytest.mark.parametrize("seqs,Hq,Hkv,D", [
    ([(300, 5000), (1, 1700), (129, 6000)], 8, 4, 128),
    ([(200, 6000), (130, 4000)], 8, 4, 64),
    ([(1900, 1900), (64, 64), (1500, 2500), (127, 127)], 32, 4, 128),
])
def test_packed_window_modes(seqs, Hq, Hkv, D, mode):
    q, k, v, cu_q, cu_k = _packed_inputs(97, seqs, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    kw, windows = MODES[mode](Hkv, 64, 1500)
    o, lse = _run_varlen(q, k, v, cu_q, cu_k, cowa.make_params(softmax_scale=scale, **kw))
    cowa.cowa_check_device_status()
    f = cowa_inputs.to_f64
    for b, (nq, nk) in enumerate(seqs):
        qs, ks = slice(cu_q[b], cu_q[b + 1]), slice(cu_k[b], cu_k[b + 1])
        rows = np.unique(np.clip([0, 1, 63, 126, 127, 128, nq - 2, nq - 1], 0, nq - 1))
        for h in range(0, Hq, Hq // 4):
            o_ref, lse_ref = orc.forward_rows(f(q[:, qs]), f(k[:, ks]), f(v[:, ks]), windows(nk), scale, h, rows)
            check(f"lse[{b},{h}]", lse[h, qs].cpu().numpy()[rows], lse_ref, TOL_LSE, TOL_LSE)
            check(f"o[{b},{h}]", o[h, qs].float().cpu().numpy()[rows], o_ref)


@pytest.mark.parametrize("B,Nq,Tmax,Hq,Hkv,D,sink,local,lens,page", [
    (1, 20, 3000, 8, 2, 128, 16, 100, [2999], None),      # 80 of 128 rows
    (2, 40, 2500, 16, 2, 128, 64, 300, [2500, 40], 64),   # three row tiles, the last half full; len = Nq
    (1, 64, 1500, 8, 8, 64, 0, 33, [1500], None),         # one head per group
    (1, 1, 30000, 2, 1, 64, 4, 64, [29999], 16),          # one unit over every block: hundreds of pieces
    (5, 3, 700, 8, 4, 128, 16, 64, [700, 3, 64, 65, 333], 80),  # lengths around one key tile, odd page size
])
def test_decode_tiles(B, Nq, Tmax, Hq, Hkv, D, sink, local, lens, page):
    multi_case(B, Nq, Tmax, Hq, Hkv, D, sink, local, lens, page_size=page)


def test_decode_of_many_sequences():
    B = 8200  # dozens of units per thread of the share-out
    multi_case(B, 1, 64, 2, 1, 64, 4, 16, [1 + i % 64 for i in range(B)], page_size=16)


@pytest.mark.parametrize("Nq,page", [(4, None), (1, 64)])
def test_decode_tiles_round_weights_below_an_exact_maximum(Nq, page):
    """The error against 64 bits is no larger than that of exact arithmetic whose weights are rounded to bf16 below the
    exact maximum of every 256 visible keys, as the single-token kernel rounds them (2 % for the fp32 sums and for which
    keys share a maximum; a reference that lags by up to 2^8 is off by 6 % more)."""
    B, Tmax, Hq, Hkv, D, sink, local = 6, 8192, 16, 8, 64, 64, 6000  # about twenty steps per block
    lens = [8192, 8000, 7777, 8100, 8191, 7900]
    q = cowa_inputs.make_train_inputs(95, B, Nq, Hq, Hkv, D)[0].permute(0, 2, 1, 3).contiguous()
    _, kc, vc, _ = cowa_inputs.make_decode_inputs(96, B, Tmax, Hq, Hkv, D, Tmax, Tmax)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale)
    o = torch.full_like(q, float("nan")).to(DEV)
    ws = torch.empty(cowa.cowa_decode_multi_workspace_bytes(B, Nq, Tmax, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
    lens_d = torch.tensor(lens, dtype=torch.int32, device=DEV)
    if page is None:
        cowa.cowa_decode_multi(q.to(DEV), kc.to(DEV), vc.to(DEV), lens_d, o, None, params, ws)
    else:
        n = Tmax // page
        table = torch.arange(B * n, dtype=torch.int32, device=DEV).reshape(B, n)
        pages = lambda x: x.reshape(B, Hkv, n, page, D).transpose(1, 2).reshape(B * n, Hkv, page, D).to(DEV)  # noqa: E731
        cowa.cowa_decode_paged(q.to(DEV), pages(kc), pages(vc), table, lens_d, o, None, params, ws)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    f = cowa_inputs.to_f64
    bf16 = lambda x: torch.from_numpy(x).to(torch.bfloat16).double().numpy()  # noqa: E731
    err = bound = 0.0
    for b in range(B):
        n, ws_ = lens[b], orc.default_windows(lens[b], Hkv, sink, local)
        want, _ = orc.forward(f(q[b].permute(1, 0, 2)), f(kc[b, :, :n]), f(vc[b, :, :n]), ws_, scale)
        err += np.sum((f(o[b].permute(1, 0, 2)) - want) ** 2)
        for h in range(Hq):
            k, v, (s, near, gap, width) = f(kc[b, h * Hkv // Hq, :n]), f(vc[b, h * Hkv // Hq, :n]), ws_[h * Hkv // Hq]
            for t in range(Nq):
                d = n - Nq + t - np.arange(n)
                seen = (d >= 0) & ((d < near) | (np.arange(n) < s) | ((d >= near + gap) & (d < near + gap + width)))
                x, vs = k[seen] @ f(q[b, t, h]) * scale, v[seen]
                acc, total = 0.0, 0.0
                for i in range(0, len(x), 256):
                    w = np.exp(x[i:i + 256] - x[i:i + 256].max())
                    up = np.exp(x[i:i + 256].max() - x.max())
                    acc, total = acc + up * (bf16(w) @ vs[i:i + 256]), total + up * w.sum()
                bound += np.sum((bf16(acc / total) - want[h, t]) ** 2)
    assert err <= 1.02 ** 2 * bound
