"""Where the kernels order the requests themselves and where the scheduler kernel does: same results on both sides of the line."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs
from gpu_utils import run_library, assert_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("io,d", [("bf16", 128), ("f32", 64)])
@pytest.mark.parametrize("n", [2, 32, 33, 64, 65])
@pytest.mark.parametrize("hv", [1, 6])
def test_order_of_requests(io, d, n, hv):
    """One and two lengths per lane, the last place of each, one request beyond; equal lengths and empty requests among them;
    37 chains and fewer run as clusters."""
    rng = np.random.default_rng(2608030310 + 100 * n + hv)
    lens = [int(x) for x in rng.integers(0, 4, size=n) * 47]
    lens[-1] = 200
    inp = make_inputs(lens, 1, hv, d, d, io, seed=90_000 + n)
    o, st, launches = run_library(inp, canary=True)
    assert launches == (1 if n <= 64 else 2)
    ro, rst = oracle.gdn_forward_inputs(inp)
    assert_parity(inp, o, st, ro, rst)
    o2, st2, launches = run_library(inp, fn="gdn_tail_replay_static_scratch")    # always from the scheduler kernel's list
    assert launches == 2
    np.testing.assert_allclose(o2, o, rtol=0, atol=0)
    np.testing.assert_allclose(st2, st, rtol=0, atol=0)


@pytest.mark.parametrize("io,d", [("bf16", 128), ("f32", 64)])
def test_more_items_than_a_cta_keeps_in_its_table(io, d):
    """5,000 short requests x 2 heads: 68 rounds of chains on 148 SMs, past the 64 that a CTA of the tensor-core kernel looks up at its
    start."""
    lens = [int(x) for x in np.random.default_rng(77).integers(0, 4, size=5000)]
    inp = make_inputs(lens, 1, 2, d, d, io, seed=91_000)
    o, st, launches = run_library(inp, canary=True)
    assert launches == 2
    assert_parity(inp, o, st, *oracle.gdn_forward_inputs(inp))
