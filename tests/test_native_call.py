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
