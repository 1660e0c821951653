"""GPU tests of the reproducible mode's bits: gradients that repeat from run to run also have to repeat from version to version
of the kernels, so that a resumed training run goes on as it would have."""
import zlib

import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa

pytestmark = pytest.mark.gpu
DEV = "cuda"


def test_partial_dq_is_the_rounded_product_rounded_to_an_integer():
    """Every query sees its own key only, with weight one: dQ = scale x dS x K, one product per element, taken to units of
    2^-18.  Bit for bit: the product rounded to fp32, then that rounded to an integer.  One rounding for both differs."""
    B, T, Hq, Hkv, D = 1, 1024, 8, 2, 128
    scale = cowa_inputs.softmax_scale(D)
    _, k, v, d_o = cowa_inputs.make_train_inputs(360, B, T, Hq, Hkv, D)
    d_o = (d_o * 2).to(torch.bfloat16)
    v.zero_()[..., 0] = 1
    q, o, lse = torch.zeros_like(d_o), torch.zeros_like(d_o), torch.zeros(B, Hq, T)
    params = cowa.make_params(windows=[(0, 1, 0, 0)] * Hkv, softmax_scale=scale, deterministic=True)
    dev = [x.to(DEV) for x in (q, k, v, o, lse, d_o, q, k, v)]
    ws = torch.empty(cowa.cowa_bwd_workspace_bytes(B, T, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
    cowa.cowa_bwd(*dev, params, ws)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()

    ds = d_o[..., :1].float().numpy()
    raw = ds * k.float().numpy().repeat(Hq // Hkv, axis=1)  # exact: eight bits by eight
    unit = np.float32(scale) * np.float32(2.0 ** 18)
    bf16 = lambda n: torch.from_numpy((n * 2.0 ** -18).astype(np.float32)).to(torch.bfloat16)  # noqa: E731
    want = bf16(np.rint(raw * unit))
    assert raw.dtype == np.float32 and np.abs(raw * unit).max() < 2.0 ** 22
    assert not torch.equal(want, bf16(np.rint(raw.astype(np.float64) * unit))), "these inputs do not tell the two apart"
    assert torch.equal(dev[6].cpu(), want)


# CRC-32 of dq, dk, dv on 148 SMs, from the kernels with steps of 64 queries and fixed parts of a tile.
BITS = {
    "2 x 1500": (dict(B=2, T=1500, Hq=8, Hkv=2, D=128, sink=64, local=300), ["c5f4dfc5", "61d4b0b5", "26ea0cb6"]),
    "4 x 821, D = 64": (dict(B=4, T=821, Hq=8, Hkv=2, D=64, sink=4, local=466), ["7f171c79", "e51785dd", "ae574f57"]),
    "one rank of eight": (dict(B=1, T=5001, Hq=8, Hkv=1, D=128, sink=128, local=896, hkv_global=8, hkv_offset=3),
                          ["114dc5d2", "032a15d7", "01266807"]),
    "packed": (dict(lens=[300, 1, 64, 777, 0, 129, 400], Hq=8, Hkv=2, D=128, sink=16, local=200),
               ["349c5ee9", "d4141c35", "bbbfab1a"]),
}


def gradient_bits(B=1, T=0, Hq=0, Hkv=0, D=0, lens=None, **window):
    """Gradients of random tensors: o and lse need not be the forward's, whose bits are not the subject here.  Multiples of
    1/64 from integers, so that every host draws the same."""
    rng = np.random.RandomState(370)
    n = sum(lens) if lens else T
    draw = lambda H, *D: torch.from_numpy(rng.randint(-127, 128, (B, H, n, *D)) / np.float32(64))  # noqa: E731
    q, d_o, o = (draw(Hq, D).to(torch.bfloat16) for _ in range(3))
    k, v = (draw(Hkv, D).to(torch.bfloat16) for _ in range(2))
    lse = draw(Hq).float() + 4
    if lens:
        q, k, v, d_o, o, lse = (x[0] for x in (q, k, v, d_o, o, lse))
    q, k, v, d_o, o, lse = (x.to(DEV) for x in (q, k, v, d_o, o, lse))
    params = cowa.make_params(softmax_scale=cowa_inputs.softmax_scale(D), deterministic=True, **window)
    grads = [torch.full_like(x, float("nan")) for x in (q, k, v)]
    if lens:
        n = cowa.cowa_bwd_varlen_workspace_bytes(len(lens), sum(lens), Hq, Hkv, D, params)
        cu = torch.tensor(np.cumsum([0] + lens), dtype=torch.int32, device=DEV)
        ws = torch.empty(n, dtype=torch.uint8, device=DEV)
        cowa.cowa_bwd_varlen(q, k, v, o, lse, d_o, *grads, cu, params, ws)
    else:
        ws = torch.empty(cowa.cowa_bwd_workspace_bytes(B, T, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
        cowa.cowa_bwd(q, k, v, o, lse, d_o, *grads, params, ws)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    return ["%08x" % zlib.crc32(x.cpu().view(torch.int16).numpy().tobytes()) for x in grads]


@pytest.mark.parametrize("name", BITS)
def test_gradients_have_the_bits_that_they_always_had(name):
    case, want = BITS[name]
    assert gradient_bits(**case) == want
