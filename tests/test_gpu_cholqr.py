"""Double-float block orthonormalisation: Cholesky QR and the panels it leaves to Gram-Schmidt."""
import numpy as np
import pytest

from paper_1904_08678_gb300 import inputs
from tests.gpu_util import dev, host, rel

pytestmark = pytest.mark.gpu


def q_factor(dims, block, nvec, vecs, df, level=0):
    from paper_1904_08678_gb300 import wcmg
    if level == 0:
        p = wcmg.default_params(dims=dims, blocks=[block], nvec=[nvec], ortho_df=df)
    else:  # a coarse level of `dims` sites with 6 components
        fine = [2 * d for d in dims]
        p = wcmg.default_params(dims=fine, n_levels=3, blocks=[(2, 2, 2, 2), block], nvec=[3, nvec], ortho_df=df)
    ctx = wcmg.Context(p)
    ctx.set_nullvecs(level, dev(vecs))
    out = dev(np.full(vecs.shape, np.nan, dtype=complex))
    ctx.get_nullvecs(level, out)
    return host(out)


# column counts around the 3 x 3 blocks and the groups of 4; panels of less than one tile,
# a ragged last tile, 1536 and 2048 rows
CASES = [((2, 4, 2, 2), (1, 2, 1, 1), 1), ((4, 2, 2, 2), (2, 1, 1, 1), 2), ((2, 2, 3, 3), (2, 2, 3, 3), 3),
         ((4, 4, 4, 4), (2, 2, 2, 2), 4), ((6, 3, 3, 3), (3, 3, 3, 3), 23), ((4, 4, 4, 8), (4, 4, 4, 4), 24),
         ((4, 4, 4, 4), (4, 4, 4, 2), 25), ((4, 4, 4, 5), (4, 4, 4, 5), 32)]


@pytest.mark.parametrize("dims,block,nvec", CASES)
def test_same_factor_as_fp64_gram_schmidt(dims, block, nvec):
    """The positive-diagonal Q factor is unique; both agree to a few hundred units of 2^-48."""
    v = inputs.complex_gaussian(31, nvec, (nvec, int(np.prod(dims)), 4, 3))
    v[nvec // 2:] += 0.5 * v[0]
    assert rel(q_factor(dims, block, nvec, v, 1), q_factor(dims, block, nvec, v, 0)) < 1e-12


def test_coarse_level_layout():
    dims, block, nvec = (4, 2, 4, 6), (2, 2, 2, 3), 5
    v = inputs.complex_gaussian(32, 1, (nvec, int(np.prod(dims)), 6))
    assert rel(q_factor(dims, block, nvec, v, 1, level=1), q_factor(dims, block, nvec, v, 0, level=1)) < 1e-12


def test_ill_conditioned_aggregate_among_good_ones():
    """One aggregate's columns nearly parallel (condition 1e4 and more): its panels go to
    Gram-Schmidt (error condition x 1e-14, columns orthonormal), its neighbours do not."""
    dims, block, nvec = (4, 4, 4, 4), (2, 2, 2, 2), 6
    v = inputs.complex_gaussian(33, 1, (nvec, 4, 4, 4, 4, 4, 3))
    bad = (slice(None), slice(0, 2), slice(2, 4), slice(0, 2), slice(2, 4))
    w = v[bad]
    v[bad] = w[:1] + 1e-4 * w
    v = v.reshape(nvec, 256, 4, 3)
    a, b = q_factor(dims, block, nvec, v, 1), q_factor(dims, block, nvec, v, 0)
    a, b = (q.reshape((nvec, 4, 4, 4, 4, 4, 3)) for q in (a, b))
    assert rel(a[bad], b[bad]) < 1e-9
    panel = a[bad].reshape(nvec, -1, 4, 3)
    for s in (slice(0, 2), slice(2, 4)):
        q = panel[:, :, s].reshape(nvec, -1)
        assert np.abs(q.conj() @ q.T - np.eye(nvec)).max() < 1e-13
    a[bad], b[bad] = 0, 0
    assert rel(a, b) < 1e-12


def test_rank_deficient_aggregate_is_refused():
    from paper_1904_08678_gb300 import wcmg
    v = inputs.complex_gaussian(34, 1, (3, 256, 4, 3))
    v[2] = 0
    ctx = wcmg.Context(wcmg.default_params(dims=(4, 4, 4, 4), blocks=[(2, 2, 2, 2)], nvec=[3], ortho_df=1))
    with pytest.raises(wcmg.WcmgError) as e:
        ctx.set_nullvecs(0, dev(v))
    assert e.value.code == wcmg.ERR_NAN


def chained_panels(nvec, keep):
    """One 4^4 aggregate, 1536 rows per chirality: unit columns a_j = keep q_j + sqrt(1 - keep^2) q_{j-1}
    with orthonormal q.  Every pivot is about keep^2 or more; the condition number grows
    geometrically with the columns."""
    R = np.diag(np.full(nvec, keep)) + np.diag(np.full(nvec - 1, np.sqrt(1 - keep**2)), 1)
    R[0, 0] = 1
    out = np.empty((nvec, 256, 2, 6), complex)
    for s in (0, 1):
        q, _ = np.linalg.qr(inputs.complex_gaussian(35 + s, nvec, (1536, nvec)))
        out[:, :, s] = (q @ R).T.reshape(nvec, 256, 6)
    return out.reshape(nvec, 256, 4, 3), np.linalg.cond(R)


# The double-float unit here is 1e-14 (the factor of a well-conditioned panel): twice that times
# the condition number, on panels that Cholesky QR takes (0.95 to 0.8) and on such as it
# must leave (0.6 and less; its own error there is the square of the condition number).
@pytest.mark.parametrize("nvec,keep", [(24, 0.95), (32, 0.9), (24, 0.8), (32, 0.8), (24, 0.6), (32, 0.6), (24, 0.53),
                                       (8, 0.283), (10, 0.283), (4, 0.28)])
def test_chained_columns_stay_orthonormal(nvec, keep):
    v, cond = chained_panels(nvec, keep)
    a, b = q_factor((4, 4, 4, 4), (4, 4, 4, 4), nvec, v, 1), q_factor((4, 4, 4, 4), (4, 4, 4, 4), nvec, v, 0)
    for s in (0, 1):
        q = a.reshape(nvec, 256, 2, 6)[:, :, s].reshape(nvec, -1)
        assert np.abs(q.conj() @ q.T - np.eye(nvec)).max() < 2e-14 * cond
    assert rel(a, b) < 2e-14 * cond


@pytest.mark.parametrize("nvec,keep", [(32, 0.8), (24, 0.75), (24, 0.6), (10, 0.283)])
def test_chained_columns_from_fp32(nvec, keep):
    """The set-up's FP32 vectors (no sweeps): the same bound for the factor of the rounded columns,
    whose condition number the rounding changes by less than 1e-6 x condition."""
    from paper_1904_08678_gb300 import wcmg
    dims, block = (4, 4, 4, 8), (4, 4, 4, 4)
    v, cond = chained_panels(nvec, keep)
    v = np.concatenate([v, v[:, ::-1]], axis=1).astype(np.complex64).astype(complex)  # two aggregates along t
    ctx = wcmg.Context(wcmg.default_params(dims=dims, blocks=[block], nvec=[nvec], ortho_df=1, inner_prec=wcmg.F32,
                                           setup_init_sweeps=0, setup_refine_sweeps=0))
    ctx.set_gauge(dev(inputs.random_gauge(dims, 0.3, 36)))
    ctx.setup(dev(v))
    out = dev(np.full(v.shape, np.nan, dtype=complex))
    ctx.get_nullvecs(0, out)
    a, b = host(out), q_factor(dims, block, nvec, v, 0)
    for q in (a.reshape(nvec, 2, 256, 2, 6)[:, i, :, s].reshape(nvec, -1) for i in (0, 1) for s in (0, 1)):
        assert np.abs(q.conj() @ q.T - np.eye(nvec)).max() < 2e-14 * cond
    assert rel(a, b) < 2e-14 * cond
