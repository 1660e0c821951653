"""GPU tests of the backward's 128-query steps where they can go wrong: sequences that end in the first or second half of a
step (the row space is padded to 64 rows only, and what lies behind it is not zero), one step, several; and the two ways in
which the reproducible mode rounds a partial dQ to an integer."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from oracle import cowa_oracle as orc

pytestmark = pytest.mark.gpu
DEV = "cuda"


def run_bwd(q, k, v, d_o, params, packed=None):
    """Gradients of one call whose workspace holds NaN before it; packed: lengths of the sequences of a packed batch."""
    qd, kd, vd, dod = (x.to(DEV) for x in (q, k, v, d_o))
    o = torch.empty_like(qd)
    lse = torch.empty(qd.shape[:-1], dtype=torch.float32, device=DEV)
    dq, dk, dv = (torch.full_like(x, float("nan")) for x in (qd, kd, vd))
    if packed is None:
        cowa.cowa_fwd(qd, kd, vd, o, lse, params)
        B, Hq, T, D = qd.shape
        ws = torch.full((cowa.cowa_bwd_workspace_bytes(B, T, Hq, kd.shape[1], D, params),), 0xFF, dtype=torch.uint8, device=DEV)
        cowa.cowa_bwd(qd, kd, vd, o, lse, dod, dq, dk, dv, params, ws)
    else:
        cu = torch.tensor(np.cumsum([0] + packed), dtype=torch.int32, device=DEV)
        cowa.cowa_prefill_varlen(qd, kd, vd, o, lse, cu, cu, params)
        n = cowa.cowa_bwd_varlen_workspace_bytes(len(packed), qd.shape[1], qd.shape[0], kd.shape[0], qd.shape[2], params)
        ws = torch.full((n,), 0xFF, dtype=torch.uint8, device=DEV)
        cowa.cowa_bwd_varlen(qd, kd, vd, o, lse, dod, dq, dk, dv, cu, params, ws)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    return [x.float().cpu().numpy() for x in (dq, dk, dv)]


def check(name, got, want, unit=1.0):
    """The suite's gradient bound, max-abs 2e-2 and half a bf16 ulp of the value; `unit`: gradients are linear in dO."""
    assert np.isfinite(got).all(), name
    assert (np.abs(got - want) - 2.0 ** -8 * np.abs(want)).max() <= 2e-2 * unit, f"{name}: {np.abs(got - want).max():.3e}"


@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("T", [1, 63, 64, 65, 128, 129, 192, 193, 577])
def test_sequence_ends_anywhere_in_a_step(T, D, deterministic):
    Hq, Hkv, sink, local = 4, 2, 7, 50
    q, k, v, d_o = cowa_inputs.make_train_inputs(310 + T, 1, T, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale, deterministic=deterministic)
    f = cowa_inputs.to_f64
    want = orc.backward(f(q[0]), f(k[0]), f(v[0]), f(d_o[0]), orc.default_windows(T, Hkv, sink, local), scale)
    for n, a, b in zip(("dq", "dk", "dv"), run_bwd(q, k, v, d_o, params), want):
        check(n, a[0], b)


@pytest.mark.parametrize("D", [64, 128])
def test_packed_sequences_end_anywhere_in_a_step(D):
    lens, Hq, Hkv, sink, local = [64, 1, 129, 192, 65, 320, 127], 4, 2, 5, 40
    total = sum(lens)
    q, k, v, d_o = (x[0] for x in cowa_inputs.make_train_inputs(330, 1, total, Hq, Hkv, D))
    scale = cowa_inputs.softmax_scale(D)
    got = run_bwd(q, k, v, d_o, cowa.make_params(sink=sink, local=local, softmax_scale=scale), packed=lens)
    f, r0 = cowa_inputs.to_f64, 0
    for T in lens:
        r = slice(r0, r0 + T)
        want = orc.backward(f(q[:, r]), f(k[:, r]), f(v[:, r]), f(d_o[:, r]), orc.default_windows(T, Hkv, sink, local), scale)
        for n, a, b in zip(("dq", "dk", "dv"), got, want):
            check(f"{n} of {T}", a[:, r], b)
        r0 += T


@pytest.mark.parametrize("unit", [1.0, 64.0])
def test_reproducible_mode_rounds_small_and_large_partial_sums_alike(unit):
    """Partial dQ below 16 take the short way, larger ones the two-part one; 64 dO puts both into one call."""
    T, Hq, Hkv, D, sink, local = 300, 4, 2, 128, 7, 120
    q, k, v, d_o = cowa_inputs.make_train_inputs(340, 1, T, Hq, Hkv, D)
    d_o = d_o * unit
    scale = cowa_inputs.softmax_scale(D)
    f = cowa_inputs.to_f64
    want = orc.backward(f(q[0]), f(k[0]), f(v[0]), f(d_o[0]), orc.default_windows(T, Hkv, sink, local), scale)
    assert (np.abs(want[0]).max() > 32) == (unit > 1)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale, deterministic=True)
    first = run_bwd(q, k, v, d_o, params)
    for n, a, b in zip(("dq", "dk", "dv"), first, want):
        check(n, a[0], b, unit)
    for a, b in zip(first, run_bwd(q, k, v, d_o, params)):
        assert np.array_equal(a, b)
