"""The fixed launch rule of the one-rhs coarse apply on lattices on both sides of two sites per SM:
integer links and vectors, so every shape must give the oracle's result bit for bit."""
import numpy as np
import pytest

from oracle.coarse import CoarseOperator
from oracle.lattice import coarse_dims, to_grid
from tests.gpu_util import dev, fields, host

pytestmark = pytest.mark.gpu


SMALL = [((6, 6, 4, 8), 1), ((8, 8, 8, 8), 3), ((8, 8, 8, 16), 6), ((8, 8, 12, 16), 5)]
CASES = [(d, n, k) for d, n in SMALL for k in ("F32", "BF16", "F16", "F64")]
CASES += [((8, 8, 8, 16), 32, "F32"), ((8, 8, 16, 16), 32, "BF16")]  # 151 MB of links: more than L2 keeps


@pytest.mark.parametrize("dims,nvec,links", CASES)
def test_default_rule_is_exact(lib, dims, nvec, links):
    block = (2, 2, 2, 2)
    cd, nb = coarse_dims(dims, block), 2 * nvec
    Vc = int(np.prod(cd))
    rng = np.random.default_rng(17)
    A = (rng.integers(-3, 4, size=(9, Vc, nb, nb)) + 1j * rng.integers(-3, 4, size=(9, Vc, nb, nb))).astype(complex)
    prec = lib.F64 if links == "F64" else lib.F32
    ctx = lib.Context(lib.default_params(dims=dims, blocks=[block], nvec=[nvec], max_rhs=1, inner_prec=prec,
                                         coarse_link_prec=lib.F32 if links == "F64" else getattr(lib, links)))
    ctx.set_coarse_links(1, dev(A))
    op = CoarseOperator(np.stack([to_grid(A[d], cd) for d in range(9)]), cd)
    phi = (rng.integers(-2, 3, size=(1, Vc, nb)) + 1j * rng.integers(-2, 3, size=(1, Vc, nb))).astype(complex)
    out = dev(np.zeros_like(phi))
    ctx.apply_coarse(1, dev(phi), out, prec=prec)
    assert np.array_equal(host(out)[0], op(fields(phi, cd, nb)[0]).reshape(Vc, nb))
