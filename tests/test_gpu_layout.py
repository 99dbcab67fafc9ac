"""External <-> internal field layout at the edges of the conversion kernels' site tiles."""
import numpy as np
import pytest

from tests.gpu_util import dev, ext, fields, host, rel
from oracle.wilson import WilsonClover

pytestmark = pytest.mark.gpu


# one site, one site short of / exactly / one row over the 128-site tile, a ragged last tile
@pytest.mark.parametrize("dims", [(1, 1, 1, 1), (1, 1, 1, 127), (4, 4, 4, 2), (3, 1, 1, 43), (5, 3, 7, 3)])
@pytest.mark.parametrize("nrhs,prec,tol", [(1, "F64", 1e-13), (3, "F64", 1e-13), (1, "F32", 3e-6), (5, "F32", 3e-6)])
def test_operator_round_trip(dims, nrhs, prec, tol):
    """pack, D, unpack against the oracle: 1872 flops per site at unit roundoff 6e-8 (FP32)."""
    from paper_1904_08678_gb300 import inputs, wcmg
    V = int(np.prod(dims))
    U = inputs.random_gauge(dims, 0.3, 7)
    b = inputs.source(dims, 3, nrhs)
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[(1, 1, 1, 1)], nvec=[2], m0=-0.1, csw=1.0, max_rhs=5))
    ctx.set_gauge(dev(U))
    x = dev(np.zeros_like(b))
    ctx.apply_D(dev(b), x, nrhs, getattr(wcmg, prec))
    D = WilsonClover(U, dims, -0.1, 1.0)
    want = ext([D(f) for f in fields(b, dims, 12)]).reshape(nrhs, V, 4, 3)
    assert rel(host(x).reshape(nrhs, V, 4, 3), want) < tol


# The last rhs count that all run at once (152 CTAs of 128 sites: stored directly) and the first that
# does not (through shared memory), with the same ragged tiles.
@pytest.mark.parametrize("dims,nrhs", [((1, 1, 1, 127), 152), ((1, 1, 1, 127), 153), ((3, 1, 1, 43), 76),
                                       ((3, 1, 1, 43), 77), ((4, 4, 4, 2), 153), ((5, 3, 7, 3), 51), ((1, 1, 1, 1), 153)])
@pytest.mark.parametrize("prec,tol", [("F64", 1e-13), ("F32", 3e-6)])
def test_round_trip_of_many_fields(dims, nrhs, prec, tol):
    from paper_1904_08678_gb300 import inputs, wcmg
    V = int(np.prod(dims))
    U = inputs.random_gauge(dims, 0.3, 8)
    b = inputs.complex_gaussian(8, 1, (nrhs, V, 4, 3))
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[(1, 1, 1, 1)], nvec=[2], m0=-0.1, csw=1.0, max_rhs=nrhs))
    ctx.set_gauge(dev(U))
    x = dev(np.full_like(b, np.nan))
    ctx.apply_D(dev(b), x, nrhs, getattr(wcmg, prec))
    D = WilsonClover(U, dims, -0.1, 1.0)
    want = ext([D(f) for f in fields(b, dims, 12)]).reshape(nrhs, V, 4, 3)
    assert rel(host(x).reshape(nrhs, V, 4, 3), want) < tol
