"""fp32 path, many requests that do not fill a block of eight tokens on average: the instance made for them, on both sides of its line."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs
from gpu_utils import run_library, assert_parity, simt_instance, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("dk,dv", [(64, 64), (128, 64), (64, 128), (128, 128)])
@pytest.mark.parametrize("lens", [[1] * 70, list(range(1, 9)) * 9, [0, 1, 2, 9, 17, 3] * 12, [8] * 70, [8] * 69 + [9]])
def test_short_requests(dk, dv, io, lens):
    """70 requests x 2 heads are more than 48 rows of values per SM on a 148-SM device at dv = 64 too."""
    inp = make_inputs(lens, 1, 2, dk, dv, io, seed=900 + dk + dv + len(lens))
    st0 = np.random.default_rng(9).standard_normal((len(lens), 2, dk, dv)).astype(np.float32)
    o, st, _ = run_library(inp, kernel=1, canary=True, init_state=st0)
    assert_parity(inp, o, st, *oracle.gdn_forward_inputs(inp, init_state=st0))


@pytest.mark.parametrize("off", [0, 4])                    # floats: a state on a 32-byte boundary, and on a 16-byte one only
@pytest.mark.parametrize("n", [3, 6, 12, 20, 80])          # every instance of the kernel on a 148-SM device, that of short requests last
def test_state_buffers_of_either_alignment(n, off):
    import torch
    import paper_2608_30310_b200 as gdn
    assert simt_instance(n * 2 * 64) == {3: (1, 2, 6), 6: (1, 4, 4), 12: (2, 2, 4), 20: (4, 4, 2), 80: (8, 4, 2)}[n]
    inp = make_inputs([5 + i % 3 for i in range(n)], 1, 2, 64, 64, "f32", seed=930)
    q, k, v, g, beta, cu = to_torch(inp, "cuda")
    size = n * 2 * 64 * 64
    a, b = torch.full((size + 16,), 7.0, device="cuda"), torch.randn(size + 16, device="cuda")
    st, st0 = (x[off:off + size].view(n, 2, 64, 64) for x in (a, b))
    o = torch.empty_like(v)
    gdn.gdn_tail_replay(q, k, v, g, beta, cu, 64, o, st, kernel=1, init_state=st0)
    ro, rst = oracle.gdn_forward_inputs(inp, init_state=st0.cpu().numpy())
    assert_parity(inp, o.cpu().numpy(), st.cpu().numpy(), ro, rst)
    assert bool((a[:off] == 7.0).all()) and bool((a[off + size:] == 7.0).all())
