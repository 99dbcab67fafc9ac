"""Minimal-residual steps at every way the step count splits into pairs and single steps."""
import numpy as np
import pytest

from oracle.aggregation import Aggregation
from oracle.coarse import coarsen
from oracle.lattice import coarse_dims
from oracle.solvers import mr
from oracle.wilson import WilsonClover
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, ext, fields, host, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("prec,tol", [("F64", 1e-12), ("F32", 1e-5)])
def test_mr_steps(steps, prec, tol):
    from paper_1904_08678_gb300 import wcmg
    dims, block, nvec, nrhs = (4, 6, 2, 4), (2, 3, 2, 2), 3, 3
    U = inputs.random_gauge(dims, 0.3, 21)
    V = int(np.prod(dims))
    raw = inputs.complex_gaussian(21, 1, (nvec, V, 12))
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[block], nvec=[nvec], m0=-0.1, csw=1.0, max_rhs=nrhs,
                                           inner_prec=getattr(wcmg, prec)))
    ctx.set_gauge(dev(U))
    ctx.set_nullvecs(0, dev(raw))
    ctx.coarsen(0)
    D = WilsonClover(U, dims, -0.1, 1.0)
    D1 = coarsen(D, Aggregation(dims, block, fields(raw, dims, 12)))
    cd = coarse_dims(dims, block)
    for level, op, d, nc in ((0, D, dims, 12), (1, D1, cd, 2 * nvec)):
        b = inputs.complex_gaussian(21, 5 + level, (nrhs, int(np.prod(d)), nc))
        x = dev(np.zeros_like(b))
        ctx.krylov(level, 0, dev(b), x, nrhs, steps)
        want = ext([mr(op, f, steps) for f in fields(b, d, nc)])
        assert rel(host(x), want) < tol, level
