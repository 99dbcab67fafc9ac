"""Restriction and prolongation of one field in 16-byte pieces: odd aggregates (which keep the
element-wise kernels), aggregates below and above a warp's pieces, padded vector groups, and
vector sets on both sides of what L2 keeps."""
import numpy as np
import pytest

from oracle.aggregation import Aggregation
from oracle.lattice import coarse_dims
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, ext, fields, host, rel

pytestmark = pytest.mark.gpu

CASES = [((3, 6, 3, 3), (3, 3, 3, 3), 2), ((4, 2, 2, 4), (2, 1, 1, 2), 3), ((4, 4, 2, 4), (2, 2, 2, 4), 9),
         ((6, 4, 4, 4), (3, 4, 4, 2), 7), ((8, 4, 4, 8), (4, 4, 4, 4), 24), ((16, 16, 16, 16), (4, 4, 4, 4), 17)]


@pytest.mark.parametrize("dims,block,nvec", CASES)
def test_against_oracle(dims, block, nvec):
    """Sums of at most 1536 products of unit-norm columns: 1e-12 in FP64, 3e-6 in FP32."""
    from paper_1904_08678_gb300 import wcmg
    V = int(np.prod(dims))
    cd = coarse_dims(dims, block)
    Vc = int(np.prod(cd))
    raw = inputs.complex_gaussian(6, 1, (nvec, V, 12))
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[block], nvec=[nvec], max_rhs=1))
    ctx.set_nullvecs(0, dev(raw))
    agg = Aggregation(dims, block, fields(raw, dims, 12))
    psi = inputs.complex_gaussian(6, 2, (1, V, 12))
    phi = inputs.complex_gaussian(6, 3, (1, Vc, 2 * nvec))
    down = ext([agg.restrict(f) for f in fields(psi, dims, 12)])
    up = ext([agg.prolong(f) for f in fields(phi, cd, 2 * nvec)])
    for prec, tol in ((wcmg.F64, 1e-12), (wcmg.F32, 3e-6)):
        c = dev(np.full((1, Vc, 2 * nvec), np.nan, dtype=complex))
        ctx.restrict(0, dev(psi), c, 1, prec)
        assert rel(host(c), down) < tol, prec
        f = dev(np.full((1, V, 12), np.nan, dtype=complex))
        ctx.prolong(0, dev(phi), f, 1, prec)
        assert rel(host(f), up) < tol, prec
