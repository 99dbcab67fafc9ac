"""GMRES over restart lengths around the widths of its bookkeeping kernels (one warp per rhs, two
columns per lane), for one rhs (fused Arnoldi step) and several; the second cycle is a partial one."""
import numpy as np
import pytest

from oracle.solvers import gmres
from oracle.wilson import WilsonClover
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, ext, fields, host, rel

pytestmark = pytest.mark.gpu

DIMS, BLOCK, NVEC = (4, 6, 2, 4), (2, 3, 2, 2), 3


# Up to 67 steps' roundings, each amplified by the operator's condition number (below 100): 1e4
# roundings, 1e-12 in FP64 and 6e-4 in FP32.
@pytest.mark.parametrize("restart", [1, 8, 9, 32, 33, 64])
@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("prec,tol", [("F64", 1e-11), ("F32", 1e-3)])
def test_restart_lengths(restart, nrhs, prec, tol):
    from paper_1904_08678_gb300 import wcmg
    U = inputs.random_gauge(DIMS, 0.3, 31)
    ctx = wcmg.Context(wcmg.default_params(dims=DIMS, blocks=[BLOCK], nvec=[NVEC], m0=-0.1, csw=1.0, max_rhs=nrhs,
                                           inner_prec=getattr(wcmg, prec)))
    ctx.set_gauge(dev(U))
    D = WilsonClover(U, DIMS, -0.1, 1.0)
    b = inputs.complex_gaussian(31, 5, (nrhs, int(np.prod(DIMS)), 12))
    x = dev(np.zeros_like(b))
    iters = restart + 3
    got_its = ctx.krylov(0, 1, dev(b), x, nrhs, restart, 0.0, iters)
    sols = [gmres(D, f, restart=restart, tol=0.0, maxiter=iters) for f in fields(b, DIMS, 12)]
    assert got_its == iters
    assert rel(host(x), ext([s[0] for s in sols])) < tol
