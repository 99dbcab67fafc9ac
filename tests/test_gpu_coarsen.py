"""Galerkin operator where its route differs: links without the sigma3 symmetry keep all
nine stencils, a hermitian operator mirrors its backward blocks; column chunks and tiles."""
import numpy as np
import pytest

from oracle.aggregation import Aggregation
from oracle.coarse import CoarseOperator, coarsen
from oracle.lattice import coarse_dims, to_grid
from oracle.wilson import WilsonClover
from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, fields, host, rel

pytestmark = pytest.mark.gpu


def test_links_of_a_caller_without_symmetry():
    from paper_1904_08678_gb300 import wcmg
    dims, b0, b1, nv = (4, 8, 4, 4), (2, 2, 2, 2), (1, 2, 2, 2), (3, 5)
    cd1 = coarse_dims(dims, b0)
    V1, nb = int(np.prod(cd1)), 2 * nv[0]
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[b0, b1], nvec=list(nv), n_levels=3))
    A1 = inputs.complex_gaussian(3, 1, (9, V1, nb, nb))
    raw = inputs.complex_gaussian(3, 2, (nv[1], V1, nb))
    ctx.set_coarse_links(1, dev(A1))
    ctx.set_nullvecs(1, dev(raw))
    ctx.coarsen(1)
    cd2 = coarse_dims(cd1, b1)
    A2 = dev(np.zeros((9, int(np.prod(cd2)), 2 * nv[1], 2 * nv[1]), dtype=complex))
    ctx.get_coarse_links(2, A2)
    op = CoarseOperator(np.stack([to_grid(a.reshape(V1, -1), cd1).reshape(cd1[::-1] + (nb, nb)) for a in A1]), cd1)
    want = coarsen(op, Aggregation(cd1, b1, fields(raw, cd1, nb))).A.reshape(9, -1, 2 * nv[1], 2 * nv[1])
    assert rel(host(A2), want) < 1e-12


# two column chunks (24 + 8 vectors), coarse extents of 1 and 2; 16- and 32-column tiles
@pytest.mark.parametrize("dims,block,nvec", [((4, 4, 4, 8), (4, 4, 4, 4), 32), ((4, 2, 6, 4), (2, 2, 3, 2), 7),
                                             ((4, 6, 2, 4), (2, 3, 2, 2), 13)])
@pytest.mark.parametrize("prec,tol", [("F64", 1e-12), ("F32", 1e-5)])
def test_mirrored_blocks(dims, block, nvec, prec, tol):
    from paper_1904_08678_gb300 import wcmg
    U = inputs.random_gauge(dims, 0.35, 11)
    V, nb = int(np.prod(dims)), 2 * nvec
    raw = inputs.complex_gaussian(11, 3, (nvec, V, 12))
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[block], nvec=[nvec], m0=-0.17, csw=1.13,
                                           inner_prec=getattr(wcmg, prec)))
    ctx.set_gauge(dev(U))
    ctx.set_nullvecs(0, dev(raw))
    ctx.coarsen(0)
    A = dev(np.zeros((9, V // int(np.prod(block)), nb, nb), dtype=complex))
    ctx.get_coarse_links(1, A)
    D = WilsonClover(U, dims, -0.17, 1.13)
    want = coarsen(D, Aggregation(dims, block, fields(raw, dims, 12))).A.reshape(9, -1, nb, nb)
    assert rel(host(A), want) < tol
