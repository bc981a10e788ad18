"""Scratch of calls on several streams: each stream's is its own, and a temporary one belongs to the stream of the call."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs
from gpu_utils import assert_parity, to_torch

pytestmark = pytest.mark.gpu


def _outputs(inp, v):
    import torch
    return torch.empty_like(v), torch.empty((inp.num_seqs, inp.num_v_heads, 128, 128), device="cuda")


def test_temporary_scratch_of_a_call_on_another_stream():
    """The call is still waiting on its stream when it returns; what the current stream allocates then is not its scratch."""
    import torch
    import paper_2608_30310_b200 as gdn
    inp = make_inputs([700], 16, 32, 128, 128, "bf16", seed=950)
    q, k, v, g, beta, cu = to_torch(inp, "cuda")
    o, st = _outputs(inp, v)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        torch.cuda._sleep(50_000_000)
    gdn.gdn_tail_replay(q, k, v, g, beta, cu, 64, o, st, stream=side)
    others = [torch.full((n,), 7, dtype=torch.uint8, device="cuda") for n in (10 << 20, 9 << 20, 12 << 20, 12 << 20, 1 << 20)]
    torch.cuda.synchronize()
    assert all(bool((x == 7).all()) for x in others)
    assert_parity(inp, o.float().cpu().numpy(), st.cpu().numpy(), *oracle.gdn_forward_inputs(inp))


def test_one_workspace_on_two_streams_at_once():
    """Eight clusters each: both calls run at the same time."""
    import torch
    import paper_2608_30310_b200 as gdn
    ws = gdn.Workspace()
    work = []
    for i in range(2):
        inp = make_inputs([1500 + 300 * i], 4, 8, 128, 128, "bf16", seed=960 + i)
        x = to_torch(inp, "cuda")
        work.append((inp, x, [_outputs(inp, x[2]) for _ in range(8)], torch.cuda.Stream()))
    torch.cuda.synchronize()
    for _, _, _, s in work:
        with torch.cuda.stream(s):
            torch.cuda._sleep(5_000_000)
    for n in range(8):
        for _, x, outs, s in work:
            gdn.gdn_tail_replay(*x, 64, *outs[n], workspace=ws, stream=s)
    torch.cuda.synchronize()
    assert len({b.data_ptr() for b in ws.by_stream.values()}) == 2
    for inp, _, outs, _ in work:
        ro, rst = oracle.gdn_forward_inputs(inp)
        for o, st in outs:
            assert_parity(inp, o.float().cpu().numpy(), st.cpu().numpy(), ro, rst)


def test_a_captured_call_outlives_the_growth_of_its_workspace():
    import torch
    import paper_2608_30310_b200 as gdn
    inp = make_inputs([300], 2, 4, 128, 128, "bf16", seed=970)
    x = to_torch(inp, "cuda")
    o, st = _outputs(inp, x[2])
    ws = gdn.Workspace()
    gdn.gdn_tail_replay(*x, 64, o, st, workspace=ws)
    torch.cuda.synchronize()
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(graph, stream=side):
        gdn.gdn_tail_replay(*x, 64, o, st, workspace=ws, stream=side)
    ws.ensure(40 << 20, side)
    ws.ensure(40 << 20)
    fill = [torch.full((12 << 20,), 7, dtype=torch.uint8, device="cuda") for _ in range(4)]
    o.zero_(); st.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert all(bool((f == 7).all()) for f in fill)
    assert_parity(inp, o.float().cpu().numpy(), st.cpu().numpy(), *oracle.gdn_forward_inputs(inp))
