"""GPU tests of CUDA graphs: every form of the forward with backward and decode, captured behind whatever may come before a
call in a stream.  The first kernel of a call is launched programmatically, behind nodes that are no kernels too."""
import pytest
import torch

import cowa_inputs
import paper_2609_32704_b200 as cowa

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("before", ["nothing", "copy", "memset", "kernel", "other stream", "copy and other stream"])
@pytest.mark.parametrize("B,T,Hq,Hkv,sink,local", [
    (2, 1536, 8, 2, 16, 128),     # one head a block
    (2, 4096, 32, 8, 128, 1024),  # two heads a block, items taken over
    (1, 2000, 4, 2, 64, 1900),    # items shared by clusters
])
def test_calls_replay_behind_other_nodes(B, T, Hq, Hkv, sink, local, before):
    D = 128
    params = cowa.make_params(sink=sink, local=local, softmax_scale=cowa_inputs.softmax_scale(D), deterministic=True)
    q, k, v, d_o = cowa_inputs.make_train_inputs(440, B, T, Hq, Hkv, D, device=DEV)
    fresh = cowa_inputs.make_train_inputs(441, B, T, Hq, Hkv, D, device=DEV)
    o, lse = torch.empty_like(q), torch.empty((B, Hq, T), device=DEV)
    grads = [torch.empty_like(x) for x in (q, k, v)]
    ws = torch.empty(cowa.cowa_bwd_workspace_bytes(B, T, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
    one = q[:, :, -1].contiguous()
    out = torch.empty_like(one)
    lens = torch.tensor([T - 300 * b for b in range(B)], dtype=torch.int32, device=DEV)
    dws = torch.empty(cowa.cowa_decode_workspace_bytes(B, T, Hq, Hkv, D, params), dtype=torch.uint8, device=DEV)
    side, other = torch.cuda.Stream(), torch.cuda.Stream()

    def step():
        if "other" in before:
            other.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(other):
                v.copy_(fresh[2])
        if "copy" in before:
            q.copy_(fresh[0])
        elif before == "memset":
            o.zero_()
        elif before == "kernel":
            q.copy_(fresh[0])
            k.mul_(1)
        if "other" in before:
            torch.cuda.current_stream().wait_stream(other)
        cowa.cowa_fwd(q, k, v, o, lse, params)
        cowa.cowa_bwd(q, k, v, o, lse, d_o, *grads, params, ws)
        cowa.cowa_decode(one, k, v, lens, out, None, params, dws)

    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            step()
    torch.cuda.synchronize()
    for x, y in zip((q, k, v, d_o, one), (*fresh, fresh[0][:, :, -1])):
        x.copy_(y)
    step()
    torch.cuda.synchronize()
    results = [o, lse, *grads, out]
    want = [x.clone() for x in results]
    for x in results:
        x.zero_()
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    cowa.cowa_check_device_status()
    assert all(torch.equal(a, b) for a, b in zip(results, want))
