"""Single-token decode of batches of very different lengths against the float64 oracle: sequences of a few rows beside long ones,
lengths at the borders of a split, hundreds of splits and few; and that a sequence's bits do not depend on how long the others are."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from oracle import cowa_oracle as orc
from launched import launched
from test_gpu_parity import DEV, TOL_LSE, check

pytestmark = pytest.mark.gpu


def lengths(B, longest):
    """From one token up, the longest first or last by turns."""
    n = [max(1, longest * (i * i + 1) // (B * B)) for i in range(B)]
    n[-1] = longest
    return n[::-1] if B % 2 else n


@pytest.mark.parametrize("B,longest,Hq,Hkv,D,sink,local", [
    (2, 33000, 8, 1, 128, 64, 3000),
    (16, 30000, 16, 2, 128, 64, 3481),
    (8, 20000, 4, 2, 64, 0, 5000),
    (33, 9000, 4, 4, 64, 4, 2500),
    (127, 12000, 2, 1, 64, 16, 4000),
    (128, 12000, 2, 1, 64, 16, 4000),
    (129, 12000, 2, 1, 64, 16, 4000),
    (128, 4000, 1, 1, 64, 16, 2000),
    (129, 4000, 1, 1, 64, 16, 2000),
    (5, 60000, 2, 1, 128, 128, 151),  # one sequence has nearly all splits
])
def test_splits_by_length(B, longest, Hq, Hkv, D, sink, local):
    compare(lengths(B, longest), longest, Hq, Hkv, D, sink, local)


@pytest.mark.parametrize("B,longest,Hq,Hkv,D,sink,local,warps", [
    (8, 30000, 16, 2, 128, 64, 3481, 16),  # more than 32 splits a sequence: sixteen warps merge
    (8, 30000, 16, 4, 64, 64, 3481, 4),
    (3, 20000, 8, 8, 128, 0, 1000, 4),
    (40, 6000, 2, 1, 64, 16, 2000, 4),
])
def test_bits_do_not_depend_on_the_other_lengths(B, longest, Hq, Hkv, D, sink, local, warps):
    q, k, v, _ = cowa_inputs.make_decode_inputs(18, B, longest, Hq, Hkv, D, longest, longest)
    q, k, v = q.to(DEV), k.to(DEV), v.to(DEV)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=cowa_inputs.softmax_scale(D))
    ws = torch.empty(cowa.cowa_decode_workspace_bytes(B, longest, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
    first, results = longest * 5 // 9, []
    for others in (64, longest // 3, longest):  # the lengths of the sequences behind the first
        lens = torch.tensor([first] + [max(1, others - 17 * i) for i in range(B - 1)], dtype=torch.int32, device=DEV)
        o = torch.full((B, Hq, D), float("nan"), dtype=torch.bfloat16, device=DEV)
        lse = torch.full((B, Hq), float("nan"), device=DEV)
        kernels = launched(lambda: cowa.cowa_decode(q, k, v, lens, o, lse, params, ws))
        assert kernels[1][:2] == (f"cowa_decode_combine_kernel<{D},{warps}>", B * Hq)
        results.append((o[0], lse[0]))
    for o, lse in results[1:]:
        assert torch.equal(o, results[0][0]) and torch.equal(lse, results[0][1])


@pytest.mark.parametrize("call", ["decode", "multi", "paged"])
def test_lengths_written_by_the_kernel_before(call):
    """The calls' second kernel starts while the first one runs, and the multi-token merge reads the lengths then: other lengths
    in every call, each written by a kernel right ahead of it, and the results of calls that had the device to themselves."""
    B, Tmax, Hq, Hkv, D, page = 6, 30016, 16, 2, 128, 64
    q, k, v, _ = cowa_inputs.make_decode_inputs(19, B, Tmax, Hq, Hkv, D, Tmax, Tmax)
    q, k, v = q.to(DEV), k.to(DEV), v.to(DEV)
    params = cowa.make_params(sink=64, local=3000, softmax_scale=cowa_inputs.softmax_scale(D))
    ws = [torch.empty(n, dtype=torch.uint8, device=DEV) for n in (cowa.cowa_decode_workspace_bytes(B, Tmax, Hq, Hkv, D, params),
                                                                  cowa.cowa_decode_multi_workspace_bytes(B, 1, Tmax, Hq, Hkv, D, params))]
    n = Tmax // page
    pages = [x.reshape(B, Hkv, n, page, D).transpose(1, 2).reshape(B * n, Hkv, page, D).contiguous() for x in (k, v)]
    table = torch.arange(B * n, dtype=torch.int32, device=DEV).reshape(B, n)
    lens = torch.ones(B, dtype=torch.int32, device=DEV)

    def run(o):
        if call == "decode":
            cowa.cowa_decode(q, k, v, lens, o, None, params, ws[0])
        elif call == "multi":
            cowa.cowa_decode_multi(q[:, None], k, v, lens, o[:, None], None, params, ws[1])
        else:
            cowa.cowa_decode_paged(q[:, None], *pages, table, lens, o[:, None], None, params, ws[1])

    steps = torch.tensor([[1 + (i * 7919 + b * 12347) % Tmax for b in range(B)] for i in range(24)], dtype=torch.int32, device=DEV)
    got, want = ([torch.empty_like(q) for _ in steps] for _ in range(2))
    for x, o in zip(steps, want):
        lens.copy_(x)
        torch.cuda.synchronize()
        run(o)
        torch.cuda.synchronize()
    for x, o in zip(steps, got):
        torch.add(x, 0, out=lens)
        run(o)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("sink,local", [(128, 2 ** 31 - 1), (2 ** 31 - 1, 5), (2 ** 31 - 1, 2 ** 31 - 1)])
@pytest.mark.parametrize("short", [1, 60, 126, 127])
def test_windows_wider_than_any_sequence(short, sink, local):
    compare([30000, short] + [30000] * 6, 30000, 16, 2, 128, sink, local, check_at=(0, 1, 2))


@pytest.mark.parametrize("D", [64, 128])
def test_one_sequence_in_many_splits(D):
    compare([40000], 40000, 8, 1, D, 64, 100)


def compare(lens, longest, Hq, Hkv, D, sink, local, check_at=None):
    B = len(lens)
    q, k, v, _ = cowa_inputs.make_decode_inputs(17, B, longest, Hq, Hkv, D, longest, longest)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale)
    o = torch.full((B, Hq, D), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((B, Hq), float("nan"), device=DEV)
    ws = torch.empty(cowa.cowa_decode_workspace_bytes(B, longest, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
    cowa.cowa_decode(q.to(DEV), k.to(DEV), v.to(DEV), torch.tensor(lens, dtype=torch.int32, device=DEV), o, lse, params, ws)
    torch.cuda.synchronize()
    f = cowa_inputs.to_f64
    for b in check_at or sorted({0, min(1, B - 1), B // 2, max(B - 2, 0), B - 1}):
        n = lens[b]
        o_ref, lse_ref = orc.decode(f(q[b:b + 1]), f(k[b:b + 1, :, :n]), f(v[b:b + 1, :, :n]), np.array([n]), sink, local, scale)
        check(f"o[b={b}]", o[b:b + 1].float().cpu().numpy(), o_ref)
        check(f"lse[b={b}]", lse[b:b + 1].cpu().numpy(), lse_ref, TOL_LSE, TOL_LSE)
