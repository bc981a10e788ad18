"""The fp32 path with one row per sixteen lanes: few value rows in the call, two and four compute warps a CTA."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs, make_raw_inputs
from gpu_utils import run_library, assert_parity, simt_instance

pytestmark = pytest.mark.gpu


# Blocks and stages begun and full, empty, one token.  203: five stages of 48 tokens or seven of 32, of which three are in flight, so
# that every buffer is used again.
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("dk,dv", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("rows", [4 * 128, 8 * 128])          # either split on a 148-SM device (up to 592 and 1,184 rows)
@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("longest", [50, 203])
def test_few_rows(longest, dk, dv, rows, raw, io):
    lens = [17, 0, longest, 1] + ([170] if rows == 8 * 128 and dv == 64 else [])
    hv = max(1, rows // dv // len(lens))
    assert simt_instance(len(lens) * hv * dv) == {4 * 128: (1, 2, 6), 8 * 128: (1, 4, 4)}[rows]
    inp = (make_raw_inputs if raw else make_inputs)(lens, 1, hv, dk, dv, io, seed=880 + dk + dv + hv)
    st0 = np.random.default_rng(6).standard_normal((len(lens), hv, dk, dv)).astype(np.float32)
    o, st, _ = run_library(inp, kernel=1, canary=True, init_state=st0, raw_inputs=raw)
    if raw:
        ro, rst = oracle.gdn_forward_f64(*oracle.prologue(inp.q, inp.k, inp.g, inp.beta)[:2], inp.v,
                                         *oracle.prologue(inp.q, inp.k, inp.g, inp.beta)[2:], inp.cu_tail_lens, init_state=st0.astype(np.float64))
    else:
        ro, rst = oracle.gdn_forward_inputs(inp, init_state=st0)
    assert_parity(inp, o, st, ro, rst)
