"""The forms of the forward kernels, each at the sizes where its parts are uneven, against the float64 oracle: clusters of 2,
4 and 8 blocks, four streams in a block, one block per item with one and two buffers, two heads per block with an item shared by two blocks and
with items taken over; lists of as many steps as parts, fewer, and one more; tiles cut by the end of the sequence; strides of o, explicit
tuples, full attention and a rank's heads.  Every case names the form that it is about.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa
from launched import launched
from oracle import cowa_oracle as orc
from test_gpu_parity import DEV, TOL_LSE, check
from test_gpu_tiles import _prefill

pytestmark = pytest.mark.gpu


def kernel_name(D, packed, form):
    """form: blocks of the one-head kernel's clusters (2, 4, 8), "plain" and "one buffer", "streams", or "pair", "pair, shared item"."""
    packed = str(packed).lower()
    if isinstance(form, int):
        return f"cowa_fwd_kernel<{D},{packed},2,1,true>"
    return {"plain": f"cowa_fwd_kernel<{D},{packed},2,1,false>", "one buffer": f"cowa_fwd_kernel<{D},{packed},1,1,false>",
            "streams": f"cowa_fwd_kernel<{D},{packed},1,4,false>", "pair": f"cowa_fwd_pair_kernel<{D},{packed},0>",
            "pair, shared item": f"cowa_fwd_pair_kernel<{D},{packed},1>"}[form]


def check_form(launch, D, packed, form, items):
    """items: tiles of 128 queries x heads (packed batches: at least so many)."""
    assert launch.kernel == kernel_name(D, packed, form)
    blocks = {"pair": 0.5, "pair, shared item": 1}.get(form, form if isinstance(form, int) else 1) * items
    assert launch.blocks == blocks or packed and launch.blocks > blocks


# B, Nq, Nk, Hq, Hkv, sink, local, form at D = 64 and 128 (packed at D = 64 where it is another one)
FORMS = [
    (1, 1, 64, 1, 1, 0, 7, "plain", "plain"),  # a single step
    (1, 100, 125, 8, 4, 4, 30, "plain", "plain"),  # two steps: nothing to share
    (2, 128, 250, 4, 4, 4, 500, "plain", "plain"),  # four steps
    (1, 128, 500, 8, 4, 4, 500, 8, 8),         # eight
    (3, 300, 380, 6, 2, 4, 380, "plain", "plain"),  # 54 items of six steps ...
    (3, 300, 620, 6, 2, 4, 620, 2, "plain"),   # ... of ten: half of them is saved, which pays for a merge at D = 64
    (3, 300, 800, 6, 2, 4, 800, 2, 2),         # ... of thirteen
    (1, 100, 500, 2, 1, 64, 300, 8, 8),        # few items: as many parts as the list has steps
    (1, 128, 577, 3, 3, 5, 500, 8, 8),         # odd group: ten steps, the last of one key
    (1, 129, 1999, 4, 4, 64, 700, 8, 8),       # a second tile of one row
    (3, 500, 500, 3, 3, 4, 100, 4, "plain"),   # causal lists from nothing up: tiles with fewer steps than parts
    (2, 500, 500, 3, 3, 4, 100, 4, 4),
    (2, 700, 1400, 8, 8, 64, 300, "streams", "plain"),  # 96 items
    (2, 900, 900, 10, 5, 3, 130, "plain", "plain"),     # 160 items of one to seven steps
    (3, 700, 700, 20, 4, 64, 100, "plain", "plain"),    # 360 items, lists of different lengths
    (3, 520, 1100, 24, 8, 64, 100, "one buffer", "plain", "plain"),  # 360 items, lists alike: one buffer, two in the packed batch
    (2, 640, 2500, 10, 5, 100, 900, "streams", "pair, shared item"),  # 100 items of long lists
    (2, 600, 2500, 10, 5, 100, 900, "streams", "pair, shared item"),  # ... the last tile of 88 rows
    (2, 700, 1400, 4, 4, 64, 300, 2, 2),       # 48 items of 14 steps
    (2, 700, 1400, 4, 2, 64, 5, 2, 2),         # ... and a near window within one tile
    (2, 300, 1300, 5, 5, 64, 300, 4, 4),       # 30 items
    (1, 2300, 2300, 6, 3, 64, 2100, "streams", 2),  # 108 causal lists of up to 36 steps
    (2, 640, 4500, 9, 3, 64, 1500, "streams", 2),   # odd group, 90 items of 44 steps
    (2, 1000, 2100, 32, 8, 64, 1300, "one buffer", "pair"),  # 512 items
]


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("case", FORMS, ids=lambda c: "-".join(map(str, c[:7])))
def test_forms_match_the_oracle(D, case):
    B, Nq, Nk, Hq, Hkv, sink, local = case[:7]
    form = case[7] if D == 64 else case[8]
    items = -(-Nq // 128) * B * Hq
    q = cowa_inputs.make_train_inputs(301, B, Nq, Hq, Hkv, D)[0]
    _, k, v, _ = cowa_inputs.make_train_inputs(302, B, Nk, Hq, Hkv, D)
    scale = cowa_inputs.softmax_scale(D)
    params = cowa.make_params(sink=sink, local=local, softmax_scale=scale)
    o = torch.full_like(q, float("nan")).to(DEV)
    lse = torch.full((B, Hq, Nq), float("nan"), dtype=torch.float32, device=DEV)
    dev = [x.to(DEV) for x in (q, k, v)]
    check_form(launched(lambda: cowa.cowa_prefill(*dev, o, lse, params))[0], D, False, form, items)
    # the same as a packed batch of equal sequences: bit for bit
    pack = lambda x: x.permute(1, 0, 2, 3).reshape(x.shape[1], -1, x.shape[3]).contiguous()  # noqa: E731
    o2 = torch.full_like(pack(o), float("nan"))
    lse2 = torch.full((Hq, B * Nq), float("nan"), dtype=torch.float32, device=DEV)
    cu = [torch.from_numpy((np.arange(B + 1) * n).astype(np.int32)).to(DEV) for n in (Nq, Nk)]
    packed = [pack(x) for x in dev]
    launch = launched(lambda: cowa.cowa_prefill_varlen(*packed, o2, lse2, *cu, params))[0]
    check_form(launch, D, True, case[9] if D == 64 and len(case) > 9 else form, items)
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    assert torch.equal(pack(o), o2)
    assert torch.equal(lse.permute(1, 0, 2).reshape(Hq, -1), lse2)
    ws = orc.default_windows(Nk, Hkv, sink, local)
    f = cowa_inputs.to_f64
    for b in range(B):
        o_ref, lse_ref = orc.forward(f(q[b]), f(k[b]), f(v[b]), ws, scale)
        check(f"lse[b={b}]", lse[b].cpu().numpy(), lse_ref, TOL_LSE, TOL_LSE)
        check(f"o[b={b}]", o[b].float().cpu().numpy(), o_ref)


# What a call may ask for besides the default rule and contiguous tensors, in the forms that few shapes reach.
@pytest.mark.parametrize("mode", ["token-major", "full", "rank", "tuples"])
@pytest.mark.parametrize("B,Nq,Nk,Hq,Hkv,D,form", [
    (2, 600, 2500, 8, 4, 128, "pair, shared item"),
    (1, 1400, 1800, 9, 3, 128, "plain"),
    (2, 600, 2500, 8, 4, 64, "streams"),
    (4, 900, 1900, 24, 4, 64, "one buffer"),
    (2, 300, 1300, 5, 5, 64, 4),
])
def test_forms_and_modes(B, Nq, Nk, Hq, Hkv, D, form, mode):
    n = Nq - 1
    run = _prefill(B, Nq, Nk, Hq, Hkv, D, 64, 1500, token_major=mode == "token-major", mode="default" if mode == "token-major" else mode,
                   rows=[0, 1, 63, 127, 128, 129, n - 1, n])
    check_form(run, D, False, form, -(-Nq // 128) * B * Hq)


@pytest.mark.parametrize("step", [6.0, 7.0])
def test_one_and_two_buffers_add_up_alike_where_the_reference_moves(step):
    """A batched call with one S buffer and the packed call of the same sequences with two.  From tile to tile the scores rise by
    more than the 8 (log2) that move a row's reference, by so little more that what was summed before still counts."""
    B, Nq, Nk, Hq, Hkv, D = 3, 520, 1100, 24, 8, 64
    gen = torch.Generator().manual_seed(303)
    q, k, v = (torch.randn(B, H, n, D, generator=gen) for H, n in ((Hq, Nq), (Hkv, Nk), (Hkv, Nk)))
    q[..., 0], k[..., 0] = 8.0, -step * (torch.arange(Nk) // 64).float()
    q, k, v = (x.to(torch.bfloat16).to(DEV) for x in (q, k, v))
    params = cowa.make_params(sink=0, local=Nk, softmax_scale=cowa_inputs.softmax_scale(D))
    o, lse = torch.empty_like(q), torch.empty((B, Hq, Nq), device=DEV)
    assert launched(lambda: cowa.cowa_prefill(q, k, v, o, lse, params))[0].kernel == "cowa_fwd_kernel<64,false,1,1,false>"
    pack = lambda x: x.transpose(0, 1).reshape(x.shape[1], -1, D).contiguous()  # noqa: E731
    o2, lse2 = torch.empty_like(pack(o)), torch.empty((Hq, B * Nq), device=DEV)
    cu = [torch.arange(B + 1, dtype=torch.int32, device=DEV) * n for n in (Nq, Nk)]
    call = lambda: cowa.cowa_prefill_varlen(pack(q), pack(k), pack(v), o2, lse2, *cu, params)  # noqa: E731
    assert launched(call)[0].kernel == "cowa_fwd_kernel<64,true,2,1,false>"
    assert torch.equal(pack(o), o2) and torch.equal(lse.transpose(0, 1).reshape(Hq, -1), lse2)


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("packed", [False, True])
def test_no_sm_holds_three_blocks_of_clusters(D, packed):
    """Two hold all TMEM of an SM, and a third one would keep its cluster's other blocks waiting with what they hold: shared memory has
    to rule it out, as registers depend on the compiler."""
    q, k, v = (torch.zeros(shape, dtype=torch.bfloat16, device=DEV) for shape in ((4, 128, D), (2, 700, D), (2, 700, D)))
    o, lse = torch.empty_like(q), torch.empty((4, 128), device=DEV)
    params = cowa.make_params(sink=4, local=100, softmax_scale=cowa_inputs.softmax_scale(D))
    if packed:
        cu = [torch.tensor([0, n], dtype=torch.int32, device=DEV) for n in (128, 700)]
        kernel, _, shared = launched(lambda: cowa.cowa_prefill_varlen(q, k, v, o, lse, *cu, params))[0]
    else:
        kernel, _, shared = launched(lambda: cowa.cowa_prefill(q[None], k[None], v[None], o[None], lse[None], params))[0]
    assert kernel == f"cowa_fwd_kernel<{D},{str(packed).lower()},2,1,true>"
    assert 3 * (shared + 1024) > torch.cuda.get_device_properties(0).shared_memory_per_multiprocessor
