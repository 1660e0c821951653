"""The binding's native argument path against its Python path: the same results for every form of the arguments that is
accepted, the same refusal for every other one."""
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
import paper_2609_32704_b200.binding as binding


def outcome(fn):
    try:
        fn()
        return None
    except Exception as e:  # noqa: BLE001
        return type(e).__name__, str(e)


def test_cpu_tensors_are_refused_alike(monkeypatch):
    x = torch.zeros(1, 2, 4, 64, dtype=torch.bfloat16)
    p = cowa.make_params(softmax_scale=0.1)
    calls = [lambda: cowa.cowa_fwd(x, x, x, x, x, p), lambda: cowa.cowa_fwd(x, None, x, x, x, p),
             lambda: cowa.cowa_decode(x[0], x, x, x, x, None, p, x), lambda: cowa.cowa_prefill(x, x, x, x, x, None)]
    assert binding._call() is not binding._PythonPath, "the native argument path has not been built"
    native = [outcome(c) for c in calls]
    monkeypatch.setattr(binding, "_native", binding._PythonPath)
    assert native == [outcome(c) for c in calls]
    assert all(o is not None for o in native)


class Sub(torch.Tensor):
    pass


def forms(q, k, v, d_o):
    """(name, tensors of a forward and backward call) in layouts and types, plain ones and ones that are refused."""
    tm = lambda x: x.transpose(1, 2).contiguous().transpose(1, 2)  # noqa: E731
    yield "contiguous", (q, k, v, d_o)
    yield "token major", tuple(tm(x) for x in (q, k, v, d_o))
    yield "keys token major", (q, tm(k), tm(v), d_o)
    yield "keys of a wider buffer", (q, torch.cat([k, k], -1)[..., :64], torch.cat([v, v], -1)[..., :64], d_o)
    yield "parameters", tuple(torch.nn.Parameter(x) for x in (q, k, v, d_o))
    yield "subclass", tuple(x.as_subclass(Sub) for x in (q, k, v, d_o))
    yield "float16", tuple(x.half() for x in (q, k, v, d_o))
    yield "strided last axis", tuple(torch.stack([x, x], -1)[..., 0] for x in (q, k, v, d_o))
    yield "three axes", (q[0], k, v, d_o)
    yield "odd strides", tuple(torch.cat([x, x], -1)[..., 4:68] for x in (q, k, v, d_o))


@pytest.mark.gpu
def test_both_paths_agree(monkeypatch):
    B, T, Hq, Hkv, D = 2, 130, 4, 2, 64
    inputs = [x.cuda() for x in cowa_inputs.make_train_inputs(410, B, T, Hq, Hkv, D)]
    p = cowa.make_params(sink=5, local=30, softmax_scale=0.125, deterministic=True)
    ws = torch.empty(cowa.cowa_bwd_workspace_bytes(B, T, Hq, Hkv, D, p), dtype=torch.uint8, device="cuda")
    lens = torch.tensor([T, 77], dtype=torch.int32, device="cuda")
    dws = torch.empty(cowa.cowa_decode_workspace_bytes(B, T, Hq, Hkv, D, p), dtype=torch.uint8, device="cuda")
    native = binding._call()
    assert native is not binding._PythonPath

    def run(t):
        q, k, v, d_o = t
        out = [torch.zeros_like(q), torch.zeros(B, Hq, T, device="cuda")] + [torch.zeros_like(x) for x in (q, k, v)]
        out += [torch.zeros(B, Hq, D, dtype=torch.bfloat16, device="cuda"), torch.zeros(B, Hq, device="cuda")]
        first = q[:, :, 0].contiguous() if q.dim() == 4 else q
        said = [outcome(lambda: cowa.cowa_fwd(q, k, v, out[0], out[1], p)),
                outcome(lambda: cowa.cowa_bwd(q, k, v, out[0], out[1], d_o, *out[2:5], p, ws)),
                outcome(lambda: cowa.cowa_bwd(q, k, v, out[0], out[1], d_o, *out[2:5], p, ws[:64])),
                outcome(lambda: cowa.cowa_decode(first, k, v, lens, out[5], out[6], p, dws)),
                outcome(lambda: cowa.cowa_decode(first, k, v, lens, out[5], None, p, dws)),
                outcome(lambda: cowa.cowa_decode(first, k, v, lens.long(), out[5], None, p, dws))]
        torch.cuda.synchronize()
        cowa.cowa_check_device_status()
        return said, [x.detach().as_subclass(torch.Tensor).float().cpu() for x in out]

    accepted = 0
    for name, t in forms(*inputs):
        with torch.no_grad():
            monkeypatch.setattr(binding, "_native", native)
            a = run(t)
            monkeypatch.setattr(binding, "_native", binding._PythonPath)
            b = run(t)
        assert a[0] == b[0], name
        assert all(torch.equal(x, y) for x, y in zip(a[1], b[1])), name
        accepted += a[0][0] is None and bool(a[1][0].any())
    assert accepted >= 5


def packed_forms(q, k, v, d_o, cu):
    """(name, tensors of a packed call, offsets)"""
    plain = (q, k, v, d_o)
    yield "contiguous", plain, cu
    yield "parameters", tuple(torch.nn.Parameter(x) for x in plain), cu
    yield "subclass", tuple(x.as_subclass(Sub) for x in plain), cu
    yield "float16", tuple(x.half() for x in plain), cu
    yield "token major", tuple(x.transpose(0, 1).contiguous().transpose(0, 1) for x in plain), cu
    yield "keys of a wider buffer", (q, torch.cat([k, k], -1)[..., :64], v, d_o), cu
    yield "four axes", (q[None], k, v, d_o), cu
    yield "long offsets", plain, cu.long()
    yield "every second offset", plain, cu.repeat_interleave(2)[::2]
    yield "one offset", plain, cu[:1]


def decode_forms(q, k, v, table, lens):
    """(name, tensors of a call that decodes several tokens)"""
    yield "contiguous", (q, k, v, table, lens)
    yield "parameters", (torch.nn.Parameter(q), torch.nn.Parameter(k), torch.nn.Parameter(v), table, lens)
    yield "subclass", (q.as_subclass(Sub), k, v, table, lens.as_subclass(Sub))
    yield "float16", (q, k.half(), v.half(), table, lens)
    yield "keys token major", (q, k.transpose(1, 2).contiguous().transpose(1, 2), v, table, lens)
    yield "three axes", (q[0], k, v, table, lens)
    yield "long lengths", (q, k, v, table, lens.long())
    yield "long table", (q, k, v, table.long(), lens)
    yield "table of one axis", (q, k, v, table[0], lens)


def on_both_paths(monkeypatch, run, forms):
    """The outcomes of run(form) and the outputs that it fills in, on the native and on the Python path; how often all passed."""
    native, accepted = binding._call(), 0
    assert native is not binding._PythonPath
    for name, *form in forms:
        got = []
        for path in (native, binding._PythonPath):
            with torch.no_grad(), monkeypatch.context() as m:
                m.setattr(binding, "_native", path)
                got.append(run(*form))
            torch.cuda.synchronize()
            cowa.cowa_check_device_status()
        (said, out), (want_said, want) = got
        assert said == want_said, name
        assert all(torch.equal(a.detach().as_subclass(torch.Tensor), b.detach().as_subclass(torch.Tensor))
                   for a, b in zip(out, want)), name
        accepted += all(s is None for s in said[:-1])
    return accepted


@pytest.mark.gpu
def test_both_paths_agree_on_prefill_and_packed_calls(monkeypatch):
    T, Hq, Hkv, D = 300, 4, 2, 64
    q, k, v, d_o = [x[0].cuda() for x in cowa_inputs.make_train_inputs(411, 1, T, Hq, Hkv, D)]
    cu = torch.tensor([0, 100, 100, 230, T], dtype=torch.int32, device="cuda")
    p = cowa.make_params(sink=5, local=30, softmax_scale=0.125, deterministic=True)
    ws = torch.empty(cowa.cowa_bwd_varlen_workspace_bytes(4, T, Hq, Hkv, D, p), dtype=torch.uint8, device="cuda")

    def packed(t, cu):
        q, k, v, d_o = t
        o, lse = torch.zeros_like(q), torch.zeros(Hq, T, device="cuda")
        grads = [torch.zeros_like(x) for x in (q, k, v)]
        said = [outcome(lambda: cowa.cowa_prefill_varlen(q, k, v, o, lse, cu, cu, p)),
                outcome(lambda: cowa.cowa_bwd_varlen(q, k, v, o, lse, d_o, *grads, cu, p, ws)),
                outcome(lambda: cowa.cowa_bwd_varlen(q, k, v, o, lse, d_o, *grads, cu, p, ws[:64]))]
        return said, [o, lse, *grads]

    assert on_both_paths(monkeypatch, packed, packed_forms(q, k, v, d_o, cu)) == 3

    def prefill(t):
        q, k, v, _ = t
        q = q[:, :, -70:] if q.dim() == 4 else q
        o, lse = torch.zeros_like(q), torch.zeros(1, Hq, 70, device="cuda")
        return [outcome(lambda: cowa.cowa_prefill(q, k, v, o, lse, p)),
                outcome(lambda: cowa.cowa_prefill(q, k, v, o, lse.double(), p))], [o, lse]

    assert on_both_paths(monkeypatch, prefill, forms(*(x[None] for x in (q, k, v, d_o)))) >= 5


@pytest.mark.gpu
def test_both_paths_agree_on_decode_of_several_tokens(monkeypatch):
    B, Nq, Hq, Hkv, D, page, pages = 2, 3, 8, 2, 64, 64, 4
    T = page * pages
    _, k, v, _ = [x.cuda() for x in cowa_inputs.make_train_inputs(412, B, T, Hq, Hkv, D)]
    q = cowa_inputs.make_train_inputs(413, B, Nq, Hq, Hkv, D)[0].transpose(1, 2).contiguous().cuda()
    pool = [x.view(B, Hkv, pages, page, D).transpose(1, 2).reshape(B * pages, Hkv, page, D).contiguous() for x in (k, v)]
    table = torch.arange(B * pages, dtype=torch.int32, device="cuda").view(B, pages)
    lens = torch.tensor([T, 77], dtype=torch.int32, device="cuda")
    p = cowa.make_params(sink=5, local=30, softmax_scale=0.125)
    ws = torch.empty(cowa.cowa_decode_multi_workspace_bytes(B, Nq, T, Hq, Hkv, D, p), dtype=torch.uint8, device="cuda")

    def multi(t):
        q, k, v, _, lens = t
        o, lse = torch.zeros_like(q), torch.zeros(B, Nq, Hq, device="cuda")
        call = cowa.cowa_decode_multi
        return [outcome(lambda: call(q, k, v, lens, o, lse, p, ws)), outcome(lambda: call(q, k, v, lens, o, None, p, ws)),
                outcome(lambda: call(q, k, v, lens, o, lse, p, ws[:64]))], [o, lse]

    def paged(t):
        q, k, v, table, lens = t
        o, lse = torch.zeros_like(q), torch.zeros(B, Nq, Hq, device="cuda")
        call = cowa.cowa_decode_paged
        return [outcome(lambda: call(q, k, v, table, lens, o, lse, p, ws)),
                outcome(lambda: call(q, k, v, table, lens, o, None, p, ws)),
                outcome(lambda: call(q, k, v, table, lens, o, lse, p, ws[:64]))], [o, lse]

    assert on_both_paths(monkeypatch, multi, decode_forms(q, k, v, table, lens)) >= 3
    assert on_both_paths(monkeypatch, paged, decode_forms(q, *pool, table, lens)) >= 3
