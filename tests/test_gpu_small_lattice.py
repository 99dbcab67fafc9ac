"""The FP64 stencil on small lattices (one warp per direction): site counts that are no multiple of
a warp, and rhs counts on both sides of the line to the one-thread-per-site kernel."""
import numpy as np
import pytest

from oracle.wilson import WilsonClover
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, ext, fields, host, rel

pytestmark = pytest.mark.gpu


# sums of about 100 terms in FP64: 1e-14 relative, 1e-13 with a margin of ten
@pytest.mark.parametrize("dims,nrhs", [((2, 2, 1, 1), 1), ((3, 5, 2, 1), 3), ((4, 3, 2, 3), 2), ((4, 4, 4, 5), 1),
                                       ((8, 8, 8, 8), 7), ((8, 8, 8, 8), 8)])
def test_apply_f64(dims, nrhs):
    from paper_1904_08678_gb300 import wcmg
    U = inputs.random_gauge(dims, 0.3, 41)
    block = [4 if d == 8 else d for d in dims]
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[block], nvec=[2], m0=-0.1, csw=1.2, max_rhs=nrhs,
                                           inner_prec=wcmg.F64))
    ctx.set_gauge(dev(U))
    D = WilsonClover(U, dims, -0.1, 1.2)
    psi = inputs.complex_gaussian(41, 5, (nrhs, int(np.prod(dims)), 12))
    out = dev(np.zeros_like(psi))
    ctx.apply_D(dev(psi), out, nrhs, wcmg.F64)
    assert rel(host(out), ext([D.apply(f) for f in fields(psi, dims, 12)])) < 1e-13


# the same line in the minimal-residual step, whose sums the stencil leaves per 32 or per 128 sites
@pytest.mark.parametrize("dims,nrhs", [((3, 5, 2, 1), 3), ((8, 8, 8, 8), 7), ((8, 8, 8, 8), 8)])
def test_mr_f64(dims, nrhs):
    from oracle.solvers import mr
    from paper_1904_08678_gb300 import wcmg
    U = inputs.random_gauge(dims, 0.3, 42)
    block = [4 if d == 8 else d for d in dims]
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[block], nvec=[2], m0=-0.1, csw=1.2, max_rhs=nrhs,
                                           inner_prec=wcmg.F64))
    ctx.set_gauge(dev(U))
    D = WilsonClover(U, dims, -0.1, 1.2)
    b = inputs.complex_gaussian(42, 5, (nrhs, int(np.prod(dims)), 12))
    x = dev(np.zeros_like(b))
    ctx.krylov(0, 0, dev(b), x, nrhs, 2)
    assert rel(host(x), ext([mr(D, f, 2) for f in fields(b, dims, 12)])) < 1e-12
