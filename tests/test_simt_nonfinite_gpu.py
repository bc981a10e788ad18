"""fp32 path: what is not finite at one token leaves the tokens before it alone (and a query all others, a value all other rows)."""
import functools

import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs, make_raw_inputs
from gpu_utils import run_library, simt_instance, TOL

pytestmark = pytest.mark.gpu

LENS = [29, 40]                                            # the second request is never touched
# v-heads -> instance of the kernel on a 148-SM device
INSTANCES = {2: (1, 2, 6), 4: (1, 4, 4), 8: (2, 2, 4), 16: (4, 4, 2), 36: (8, 4, 2)}


def inputs(hv):
    return make_inputs(LENS, 2, hv, 128, 128, "f32", seed=880)


@functools.lru_cache(maxsize=None)
def untouched(hv):
    return oracle.gdn_forward_inputs(inputs(hv))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("name", ["q", "k", "v", "g", "beta"])
@pytest.mark.parametrize("token", [16, 19, 23, 28])        # first, inside and last of a block, last of the request
@pytest.mark.parametrize("hv", list(INSTANCES))
def test_earlier_tokens_are_untouched(hv, token, name, bad):
    assert simt_instance(len(LENS) * hv * 128) == INSTANCES[hv]
    inp, (ro, rst) = inputs(hv), untouched(hv)
    x = getattr(inp, name)
    x[(token, 0, 5) if x.ndim == 3 else (token, 0)] = bad
    o, st, _ = run_library(inp, kernel=1)
    tol = TOL["f32"]["o_max_abs"]
    np.testing.assert_allclose(o[:token], ro[:token], rtol=0, atol=tol)
    np.testing.assert_allclose(o[29:], ro[29:], rtol=0, atol=tol)
    np.testing.assert_allclose(st[1], rst[1], rtol=0, atol=tol)
    heads = hv // 2 if name in "qk" else 1                  # v-heads that see the value
    np.testing.assert_allclose(o[:, heads:], ro[:, heads:], rtol=0, atol=tol)
    assert not np.isfinite(o[token, 0]).all()
    if name == "q":
        np.testing.assert_allclose(o[token + 1:], ro[token + 1:], rtol=0, atol=tol)
        np.testing.assert_allclose(st, rst, rtol=0, atol=tol)
    elif name == "v":
        rows = [r for r in range(128) if r != 5]
        np.testing.assert_allclose(o[:, :, rows], ro[:, :, rows], rtol=0, atol=tol)
        np.testing.assert_allclose(st[..., rows], rst[..., rows], rtol=0, atol=tol)


def test_raw_inputs_too():
    inp = make_raw_inputs([24], 2, 2, 64, 64, "f32", seed=881)
    o0, _, _ = run_library(inp, kernel=1, raw_inputs=True)
    inp.k[21, 1, 3] = np.nan
    o, _, _ = run_library(inp, kernel=1, raw_inputs=True)
    np.testing.assert_array_equal(o[:21], o0[:21])
    assert np.isnan(o[21:, 1]).all()
