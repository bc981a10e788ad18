"""The fp32 path loses nothing against a plain fp32 evaluation of the recurrence, one token after the other."""
import numpy as np
import pytest

import oracle
from gdn_workloads import make_inputs
from gpu_utils import run_library, simt_instance

pytestmark = pytest.mark.gpu

# v-heads of a request at dv = 128 -> instance of the kernel on a 148-SM device
INSTANCES = {2: (1, 2, 6), 8: (1, 4, 4), 16: (2, 2, 4), 32: (4, 4, 2), 64: (8, 4, 2)}


def token_by_token_f32(inp):
    """Eq. 1 in fp32, every operation rounded, for one request with as many q/k heads as v heads."""
    f = np.float32
    q, k, v, b = (np.asarray(x, dtype=f) for x in (inp.q, inp.k, inp.v, inp.beta))
    a = np.exp(np.asarray(inp.g, dtype=f))
    T, H, dk = k.shape
    S, o = np.zeros((H, dk, v.shape[2]), f), np.zeros(v.shape, f)
    for t in range(T):
        kt, qt, at = k[t][:, None, :], q[t][:, None, :], a[t][:, None]
        r, p = (kt @ S)[:, 0], (qt @ S)[:, 0]
        d = b[t][:, None] * (v[t] - at * r)
        S = at[:, :, None] * S + k[t][:, :, None] * d[:, None, :]
        o[t] = at * p + d * (kt @ qt.transpose(0, 2, 1))[:, 0]
    return o, S[None]


@pytest.mark.parametrize("hv", list(INSTANCES))
@pytest.mark.parametrize("decay", ["recipe", "slow"])
def test_error_is_that_of_the_plain_recurrence(hv, decay):
    """Eight decays enter a block as one factor; their rounding must not add to that of eight single steps."""
    assert simt_instance(hv * 128) == INSTANCES[hv]
    inp = make_inputs([512], hv, hv, 128, 128, "f32", seed=860 + hv)
    if decay == "slow":
        inp.g[:] = np.random.default_rng(hv).uniform(-0.02, -0.0001, inp.g.shape)
    o, st, _ = run_library(inp, kernel=1)
    ro, rst = oracle.gdn_forward_inputs(inp)
    po, pst = token_by_token_f32(inp)
    for got, plain, ref in ((o, po, ro), (st, pst, rst)):
        assert np.linalg.norm(got - ref) <= np.linalg.norm(plain - ref)


@pytest.mark.parametrize("hv", list(INSTANCES))
def test_equal_decays_do_not_add_up(hv):
    """The same decay in every block: a rounding of its products would point the same way each time.  Independent roundings leave
    the state with some sqrt(n) of them, n = 9 per block over the 1 / (8 * 0.02) blocks that a decay of e^-0.08 a block remembers;
    the errors of delta that feed the state are allowed as much again."""
    inp = make_inputs([512], hv, hv, 128, 128, "f32", seed=870 + hv)
    inp.g[:] = -0.01
    o, st, _ = run_library(inp, kernel=1)
    _, rst = oracle.gdn_forward_inputs(inp)
    bound = 2 * np.sqrt(9 / (8 * 0.02)) * 2.0 ** -24 / np.sqrt(3)
    assert np.linalg.norm(st - rst) <= bound * np.linalg.norm(rst)
