"""The fp32 path's blocks of eight tokens, its stages of 16 and 32 (48: test_simt_few_rows_gpu.py), its splits of the value rows."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs
from gpu_utils import run_library, assert_parity, simt_instance

pytestmark = pytest.mark.gpu

LENS = [1, 7, 8, 9, 15, 16, 17, 31, 0, 33, 64, 100]       # around the block, both stages and three stages in flight


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("hv", [1, 2, 8, 16])             # rows per warp on a 148-SM device: 4, 8, 16, 16; at dv = 64: 2, 4, 8, 16
@pytest.mark.parametrize("dk,dv", [(64, 128), (128, 128), (128, 64)])
def test_block_edges(dk, dv, hv, io):
    assert 2 * simt_instance(len(LENS) * hv * dv)[0] == {1: 4, 2: 8, 8: 16, 16: 16}[hv] // (2 if dv == 64 and hv < 16 else 1)
    inp = make_inputs(LENS, 1, hv, dk, dv, io, seed=800 + hv + dk + dv)
    rng = np.random.default_rng(5)
    st0 = rng.standard_normal((len(LENS), hv, dk, dv)).astype(np.float32)
    o, st, _ = run_library(inp, kernel=1, canary=True, init_state=st0)
    assert_parity(inp, o, st, *oracle.gdn_forward_inputs(inp, init_state=st0))


def test_no_decay_and_full_decay_inside_a_block():
    """alpha = 1 and alpha = 0 (g = -inf) next to each other: the ratios of cumulative decays are products, not quotients."""
    inp = make_inputs([37], 2, 2, 64, 64, "f32", seed=841)
    inp.g[::3] = 0.0
    inp.g[5::7] = -np.inf
    o, st, _ = run_library(inp, kernel=1)
    assert_parity(inp, o, st, *oracle.gdn_forward_inputs(inp))
