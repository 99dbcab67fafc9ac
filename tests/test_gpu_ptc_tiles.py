"""PTC network forward and backward at the edges of its site tiles (32 and 128 sites)."""
import numpy as np
import pytest

from oracle.ptc import NHOP, PTC
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, fields, host, rel, rel_norm

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


# Whole-field error in the 2-norm, in unit roundoffs of 2^-24: a sum of n products of random sign
# taken in one chain is off by about 0.3 sqrt(n) of them, and an input or output here passes two
# layers of three sums of at most 36 (0.3 x 6 x sqrt(6) = 4.4) before, for the weights, chains of
# at most 32 + 8 + 3.  One chain over 256 products alone adds 4.8.
@pytest.mark.parametrize("dims,nrhs", [((8, 4, 4, 8), 1), ((4, 4, 4, 5), 3)])
def test_error_in_roundoffs(dims, nrhs):
    from paper_1904_08678_gb300 import wcmg
    V = int(np.prod(dims))
    U = inputs.random_gauge(dims, 0.3, 42)
    w = 0.05 * inputs.complex_gaussian(42, 1, (2, 12, NHOP, 4, 4))
    W1, W2 = w[0].reshape(12, 1, NHOP, 4, 4), w[1].reshape(1, 12, NHOP, 4, 4)
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[(1, 1, 1, 1)], nvec=[2], max_rhs=nrhs))
    ctx.set_gauge(dev(U))
    ctx.ptc_set_weights(dev(w.ravel()))
    r, g = (inputs.complex_gaussian(42, k, (nrhs, V, 4, 3)) for k in (2, 3))
    out, gin, gW = dev(np.zeros_like(r)), dev(np.zeros_like(r)), dev(np.zeros(3456, dtype=complex))
    ctx.ptc_forward(dev(r), out, nrhs)
    ctx.ptc_backward(dev(r), dev(g), gin, gW, nrhs)
    net, gw = PTC(U, dims), np.zeros((2, 12 * NHOP * 16), dtype=complex)
    want, back = np.empty((nrhs, V, 12), complex), np.empty((nrhs, V, 12), complex)
    for q, (fr, fg) in enumerate(zip(fields(r, dims, 12), fields(g, dims, 12))):
        o, cache = net.forward(W1, W2, fr)
        a1, a2, gr = net.backward(W1, W2, cache, fg)
        gw += np.stack([a1.ravel(), a2.ravel()])
        want[q], back[q] = o.reshape(V, 12), gr.reshape(V, 12)
    for got, ref in ((host(out), want), (host(gin), back), (host(gW), gw)):
        assert rel_norm(got.ravel(), ref.ravel()) < 4.4 * 2.0**-24
