"""The fp32 path with one row per sixteen lanes: few value rows in the call, two and four compute warps a CTA."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs, make_raw_inputs
from gpu_utils import run_library, assert_parity

pytestmark = pytest.mark.gpu

LENS = [17, 0, 50, 1]              # blocks and stages of 32 and 48 tokens begun and full, three stages in flight, empty, one token


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("dk,dv", [(64, 64), (64, 128), (128, 64), (128, 128)])
@pytest.mark.parametrize("rows", [4 * 128, 8 * 128])          # either split on a 148-SM device (up to 592 and 1,184 rows)
@pytest.mark.parametrize("raw", [False, True])
def test_few_rows(dk, dv, rows, raw, io):
    lens = LENS + [170] if rows == 8 * 128 and dv == 64 else LENS
    hv = max(1, rows // dv // len(lens))
    inp = (make_raw_inputs if raw else make_inputs)(lens, 1, hv, dk, dv, io, seed=880 + dk + dv + hv)
    st0 = np.random.default_rng(6).standard_normal((len(lens), hv, dk, dv)).astype(np.float32)
    o, st, _ = run_library(inp, kernel=1, canary=True, init_state=st0, raw_inputs=raw)
    if raw:
        ro, rst = oracle.gdn_forward_f64(*oracle.prologue(inp.q, inp.k, inp.g, inp.beta)[:2], inp.v,
                                         *oracle.prologue(inp.q, inp.k, inp.g, inp.beta)[2:], inp.cu_tail_lens, init_state=st0.astype(np.float64))
    else:
        ro, rst = oracle.gdn_forward_inputs(inp, init_state=st0)
    assert_parity(inp, o, st, ro, rst)
