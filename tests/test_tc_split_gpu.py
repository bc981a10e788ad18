"""The two forms of the tensor-core kernel: a chain split over a cluster (few chains) and one CTA per chain (many)."""
import numpy as np
import pytest

import oracle
import paper_2608_30310_b200 as gdn
from gdn_workloads import make_inputs
from gpu_utils import run_library, assert_parity, to_torch

pytestmark = pytest.mark.gpu

# lengths whose chunk counts run through the operand slots (3), the teams (3 x 3) and the ring (9 slots) of the split, with a
# remainder of one row, one short of a chunk and none; both sides of the 37-chain limit of the split
LENS = [[1], [64], [65, 191], [9 * 64, 10 * 64 + 1], [19 * 64 - 1], [0, 28 * 64 + 33, 0]]


@pytest.mark.parametrize("heads", [(1, 1), (2, 6), (37, 37), (38, 38)])
@pytest.mark.parametrize("lens", LENS)
def test_split_and_single_cta_forms(lens, heads):
    Hq, Hv = heads
    inp = make_inputs(lens, Hq, Hv, 128, 128, "bf16", seed=700 + Hv + sum(lens))
    o, st, _ = run_library(inp, kernel=2, canary=True)
    assert_parity(inp, o, st, *oracle.gdn_forward_inputs(inp))


def test_workspace_without_the_ring_gives_the_same_bits():
    """The operand ring is optional scratch: a workspace sized for the request list alone runs the single-CTA form."""
    import ctypes
    import torch
    inp = make_inputs([300, 65], 2, 4, 128, 128, "bf16", seed=731)
    o, st, _ = run_library(inp, kernel=2)
    q, k, v, g, beta, cu = to_torch(inp, "cuda")
    d = gdn.GdnDesc()
    d.num_qk_heads, d.num_v_heads, d.head_k_dim, d.head_v_dim, d.io_dtype = 2, 4, 128, 128, gdn.GDN_BF16
    d.num_seqs, d.total_tokens, d.kernel = 2, 365, gdn.GDN_KERNEL_TCGEN05
    o2, st2 = torch.empty_like(v), torch.empty((2, 4, 128, 128), device="cuda")
    ws = torch.empty(1024, dtype=torch.uint8, device="cuda")
    d.workspace, d.workspace_bytes = ws.data_ptr() + (-ws.data_ptr()) % 256, 512
    d.stream = torch.cuda.current_stream().cuda_stream
    assert gdn.workspace_size(d) > 512
    rc = gdn.load_library().gdn_tail_replay(ctypes.byref(d), q.data_ptr(), k.data_ptr(), v.data_ptr(), g.data_ptr(), beta.data_ptr(),
                                            cu.data_ptr(), 64, o2.data_ptr(), st2.data_ptr())
    assert rc == 0
    torch.cuda.synchronize()
    np.testing.assert_array_equal(o2.float().cpu().numpy(), o.astype(np.float32))
    np.testing.assert_array_equal(st2.cpu().numpy(), st.astype(np.float32))
