"""PTC network forward and backward at the edges of its site tiles (32 and 128 sites)."""
import numpy as np
import pytest

from oracle.ptc import NHOP, PTC
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, fields, host, rel

pytestmark = pytest.mark.gpu


# one tile short by one site, exactly full, one site over; odd numbers of tiles and samples
@pytest.mark.parametrize("dims,nrhs", [((1, 1, 1, 31), 1), ((2, 2, 2, 4), 3), ((3, 11, 1, 1), 2), ((3, 3, 5, 3), 1),
                                       ((2, 3, 1, 43), 5)])
def test_forward_backward(dims, nrhs):
    """FP32 against the FP64 oracle, relative 1e-5 as for the network's other tests."""
    from paper_1904_08678_gb300 import wcmg
    V = int(np.prod(dims))
    U = inputs.random_gauge(dims, 0.3, 41)
    w = 0.2 * inputs.complex_gaussian(41, 1, (2, 12, NHOP, 4, 4))
    W1, W2 = w[0].reshape(12, 1, NHOP, 4, 4), w[1].reshape(1, 12, NHOP, 4, 4)
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[(1, 1, 1, 1)], nvec=[2], max_rhs=nrhs))
    ctx.set_gauge(dev(U))
    ctx.ptc_set_weights(dev(w.ravel()))
    r, g = (inputs.complex_gaussian(41, k, (nrhs, V, 4, 3)) for k in (2, 3))
    out, gin, gW = dev(np.zeros_like(r)), dev(np.zeros_like(r)), dev(np.zeros(3456, dtype=complex))
    ctx.ptc_forward(dev(r), out, nrhs)
    ctx.ptc_backward(dev(r), dev(g), gin, gW, nrhs)
    net = PTC(U, dims)
    gw = np.zeros((2, 12, NHOP, 4, 4), dtype=complex)
    for q, (fr, fg) in enumerate(zip(fields(r, dims, 12), fields(g, dims, 12))):
        want, cache = net.forward(W1, W2, fr)
        a1, a2, gr = net.backward(W1, W2, cache, fg)
        gw[0] += a1.reshape(12, NHOP, 4, 4)
        gw[1] += a2.reshape(12, NHOP, 4, 4)
        assert rel(host(out)[q].reshape(V, 12), want.reshape(V, 12)) < 1e-5
        assert rel(host(gin)[q].reshape(V, 12), gr.reshape(V, 12)) < 1e-5
    assert rel(host(gW), gw.ravel()) < 1e-5
