"""GPU tests of the reproducible mode's bits: gradients that repeat from run to run also have to repeat from version to version
of the kernels, so that a resumed training run goes on as it would have."""
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
