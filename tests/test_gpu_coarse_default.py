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


# Every shape in the list is 12 applies on a context's first: two thread counts x four splits x two
# depths, the five rhs-tile shapes, the streaming ones that hold (FP32 7, BF16 12) and the fixed rule.
@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (8, 8, 8, 16)])
@pytest.mark.parametrize("links,count", [("F32", 29), ("BF16", 34)])
def test_one_rhs_tuning_list_stays_short(lib, dims, links, count):
    nvec, block = 24, (2, 2, 2, 2)
    Vc = int(np.prod(coarse_dims(dims, block)))
    ctx = lib.Context(lib.default_params(dims=dims, blocks=[block], nvec=[nvec], inner_prec=lib.F32,
                                         coarse_link_prec=getattr(lib, links)))
    ctx.set_coarse_links(1, dev(np.ones((9, Vc, 2 * nvec, 2 * nvec), dtype=complex)))
    t = ctx.tune_coarse(1, 1, lib.F32)
    assert t["candidates"] <= count
    assert t["us"] <= t["us_default"]
