"""FP32 restriction of four or more fields at the edges of its tiles."""
import numpy as np
import pytest

from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, host, rel

pytestmark = pytest.mark.gpu

# rhs: both sides of every tile width (4, 8, 12, 16, 24, 32, 48); vectors: each tile height,
# full and padded; aggregates: below one chunk per warp, ragged last chunk, 4^4
CASES = [((6, 4, 2, 4), (3, 2, 1, 2), 8), ((3, 6, 9, 3), (3, 3, 3, 3), 5), ((8, 4, 4, 8), (4, 4, 4, 4), 24),
         ((4, 4, 8, 2), (4, 4, 4, 2), 20), ((4, 4, 4, 4), (2, 2, 4, 4), 16), ((4, 8, 4, 4), (4, 4, 4, 4), 32)]


@pytest.mark.parametrize("dims,block,nvec", CASES)
def test_against_fp64(dims, block, nvec):
    """The FP64 kernels are pinned to the oracle elsewhere; an FP32 sum of up to 1536
    products of unit-norm columns with Gaussian fields stays below 3e-6 of the result."""
    from paper_1904_08678_gb300 import wcmg
    V, top = int(np.prod(dims)), 50
    Vc = V // int(np.prod(block))
    p = wcmg.default_params(dims=dims, blocks=[block], nvec=[nvec], max_rhs=top)
    ctx = wcmg.Context(p)
    ctx.set_nullvecs(0, dev(inputs.complex_gaussian(5, 1, (nvec, V, 4, 3))))
    psi = dev(inputs.complex_gaussian(5, 2, (top, V, 4, 3)))
    want = dev(np.zeros((top, Vc, 2 * nvec), dtype=complex))
    ctx.restrict(0, psi, want, top, wcmg.F64)
    want = host(want)
    for nrhs in (4, 5, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 48, 50):
        out = dev(np.full((nrhs, Vc, 2 * nvec), np.nan, dtype=complex))
        ctx.restrict(0, psi[:nrhs].contiguous(), out, nrhs, wcmg.F32)
        assert rel(host(out), want[:nrhs]) < 3e-6, nrhs
