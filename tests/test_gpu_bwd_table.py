"""The backward of few tiles, whose blocks are cut by the tiles' lengths from a table in the kernel's arguments: one item per block,
and more items than SMs, so that blocks take over further ones; tiles that no query sees; odd groups; strides; sums of the parts in
one launch with the conversion of dQ, and in one of their own.  Against the float64 oracle; the blocks are those of the rule as
tests/test_bwd_plan.py restates it."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from launched import launched
from oracle import cowa_oracle as orc
from test_bwd_plan import SMS, blocks_of
from test_gpu_bwd_steps import check

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("B,Nq,Nk,Hq,Hkv,D,sink,local,rank,single,finish", [
    (1, 3000, 3000, 8, 1, 128, 40, 200, (8, 3), True, True),  # rank: of so many KV heads, these from that one on
    (2, 700, 700, 3, 1, 128, 0, 64, (1, 0), True, True),      # an odd group: parts begin inside a head's steps
    (4, 1000, 1000, 16, 4, 128, 16, 200, (4, 0), False, True),  # more items than SMs: blocks take over
    (4, 1000, 1000, 16, 4, 64, 16, 200, (4, 0), False, True),
    (3, 1500, 1500, 12, 4, 128, 100, 700, (4, 0), False, True),
    (2, 4000, 4000, 9, 3, 64, 5, 1500, (3, 0), False, True),
    (1, 2500, 4500, 8, 4, 64, 0, 300, (4, 0), False, True),   # fewer queries than keys, tiles that no query sees
    (1, 7000, 7000, 12, 4, 128, 0, 100, (4, 0), False, True),
    (3, 2049, 2049, 21, 3, 64, 0, 35, (3, 0), False, False),  # sums in a launch of their own
    (1, 9358, 9358, 14, 2, 128, 0, 150, (8, 5), False, False),
])
@pytest.mark.parametrize("token_major", [False, True])
def test_gradients(B, Nq, Nk, Hq, Hkv, D, sink, local, rank, single, finish, token_major):
    q, _, _, d_o = cowa_inputs.make_train_inputs(380, B, Nq, Hq, Hkv, D)
    _, k, v, _ = cowa_inputs.make_train_inputs(381, B, Nk, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale, hkv_global=rank[0], hkv_offset=rank[1])
    windows = orc.default_windows(Nk, rank[0], sink, local)[rank[1]:rank[1] + Hkv]
    blocks, table = blocks_of(B, Nq, Nk, Hkv, Hq // Hkv, windows)
    assert table is not None and max(table) > 1 and (blocks <= SMS) == single
    put = (lambda x: x.transpose(1, 2).contiguous().to(DEV).transpose(1, 2)) if token_major else (lambda x: x.to(DEV))
    qd, kd, vd, dod = (put(x) for x in (q, k, v, d_o))
    o, lse = torch.empty_like(qd), torch.empty((B, Hq, Nq), device=DEV)
    cowa.cowa_prefill(qd, kd, vd, o, lse, params)
    dq, dk, dv = (torch.full_like(x, float("nan")) for x in (qd, kd, vd))
    nbytes = cowa.cowa_bwd_prefill_workspace_bytes(B, Nq, Nk, Hq, Hkv, D, params)
    ws = torch.full((nbytes + 64,), 0xFF, dtype=torch.uint8, device=DEV)
    kernels = launched(lambda: cowa.cowa_bwd_prefill(qd, kd, vd, o, lse, dod, dq, dk, dv, params, ws[:nbytes]))
    cowa.cowa_check_device_status()
    if torch.cuda.get_device_properties(0).multi_processor_count == SMS:
        assert [x.blocks for x in kernels if x.kernel == f"cowa_bwd_kernel<{D},false>"] == [blocks]
    assert any("cowa_bwd_finish_kernel" in x.kernel for x in kernels) == finish
    assert (ws[nbytes:] == 0xFF).all(), "the backward wrote past its workspace"
    f = cowa_inputs.to_f64
    for b in range(B):
        args = f(q[b]), f(k[b]), f(v[b]), f(d_o[b]), windows
        if Nq * Nk <= 3000 ** 2:
            for n, got, want in zip(("dq", "dk", "dv"), (dq, dk, dv), orc.backward(*args, scale)):
                check(f"{n}[{b}]", got[b].float().cpu().numpy(), want)
        elif b == B - 1:  # whole KV tiles: first, cut into most parts, last
            for tile in sorted({0, table.index(max(table)) // Hkv, len(table) // Hkv - 1}):
                cols = np.arange(tile * 128, min(tile * 128 + 128, Nk))
                for h in (0, Hkv - 1):
                    for n, got, want in zip(("dk", "dv"), (dk, dv), orc.backward_dkdv_cols(*args, scale, h, cols)):
                        check(f"{n}[{b},{h},{tile}]", got[b, h, cols].float().cpu().numpy(), want)
            assert torch.isfinite(dq).all()
