"""The Gram-Schmidt of an Arnoldi step, short and long vectors: orthogonality of the new basis vector."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


class GmresState(ctypes.Structure):
    _fields_ = [(f, ctypes.c_void_p) for f in ("H", "cs", "sn", "g", "y", "hnorm", "bnorm", "resid", "active", "jdone",
                                               "done")] + [("m", ctypes.c_int)]


def _symbol(name, R):
    """The library's C++ launchers, one per precision."""
    from paper_1904_08678_gb300 import wcmg
    lib = ctypes.CDLL(wcmg.LIB_PATH)
    return {
        "fused": lambda: getattr(lib, f"_ZN4wcmg20launch_arnoldi_fusedI{R}EEvPNS_7cplx_ofIT_E4typeExS5_xRKNS_10GmresState"
                                      "EiPKidiP11CUstream_stS5_"),
        "long": lambda: getattr(lib, f"_ZN4wcmg19launch_gram_schmidtI{R}EEiP7double2S2_PdPNS_7cplx_ofIT_E4typeEPKS7_xiixiS2_"
                                     "P11CUstream_stPKii"),
    }[name]()


# What a new basis vector keeps of the earlier ones when the step cancels all but 1e-3 of w: 16
# unit roundoffs for two passes (chains of a few hundred sums, random signs), against 1e2 and more
# if the second pass does not see the rounding of the first.  Its direction: 16 roundoffs of w.
@pytest.mark.parametrize("kind,n,nrhs", [("fused", 96, 1), ("fused", 9000, 1), ("fused", 24576, 1), ("fused", 60000, 1), ("fused", 131072, 1),
                                         ("long", 500, 2), ("long", 40001, 1), ("long", 40000, 3)])
@pytest.mark.parametrize("k", [1, 2, 4, 7, 20, 64])
@pytest.mark.parametrize("prec", ["f", "d"])
def test_new_basis_vector_is_orthogonal(kind, n, nrhs, k, prec):
    import torch
    rt, ct, unit = (torch.float32, torch.complex64, 2.0**-24) if prec == "f" else (torch.float64, torch.complex128, 2.0**-53)
    gen = torch.Generator(device="cuda").manual_seed(1000 * k + n)
    c128 = dict(dtype=torch.complex128, device="cuda")
    Q = torch.linalg.qr(torch.randn(nrhs, n, k + 1, generator=gen, **c128))[0].transpose(1, 2)  # [nrhs][k + 1][n]
    c = torch.randn(nrhs, 1, k, generator=gen, **c128)
    c = c / torch.linalg.vector_norm(c, dim=2, keepdim=True)
    V = torch.empty(k + 1, nrhs, n, dtype=ct, device="cuda")  # the basis, then the new vector
    V[:k] = Q[:, :k].transpose(0, 1)
    w = ((c @ Q[:, :k])[:, 0] + 1e-3 * Q[:, k]).to(ct).contiguous()
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    z = lambda *s: torch.zeros(*s, dtype=torch.float64, device="cuda")  # noqa: E731
    ll, i32 = ctypes.c_longlong, ctypes.c_int
    if kind == "fused":
        m = 64
        bufs = dict(H=z(2 * m * (m + 1)), cs=z(m) + 1, sn=z(2 * m), g=z(2 * (m + 1)) + 1, y=z(2 * m), hnorm=z(1),
                    bnorm=z(1), resid=z(1), active=torch.ones(1, dtype=torch.int32, device="cuda"),
                    jdone=torch.zeros(1, dtype=torch.int32, device="cuda"), done=torch.zeros(1, dtype=torch.int32, device="cuda"))
        S = GmresState(m=m, **{f: t.data_ptr() for f, t in bufs.items()})
        torch.cuda.synchronize()
        _symbol("fused", prec)(p(V), ll(n), p(w), ll(n), ctypes.byref(S), i32(k - 1), None, ctypes.c_double(0.0),
                               i32(0), None, None)
        torch.cuda.synchronize()
        v = V[k]
    else:
        h1, h2, part, np_ = z(nrhs, 2 * k), z(nrhs, 2 * k), z(2 * nrhs * 64 * 608), z(nrhs * 608)
        torch.cuda.synchronize()
        nb = _symbol("long", prec)(p(h1), p(h2), p(np_), p(w), p(V), ll(n * nrhs), i32(k), i32(k), ll(n), i32(nrhs),
                                   p(part), None, None, i32(0))
        torch.cuda.synchronize()
        norm = np_[:nrhs * nb].reshape(nrhs, nb).sum(1).sqrt()
        assert torch.allclose(norm, torch.linalg.vector_norm(w.to(torch.complex128), dim=1), rtol=100 * unit)
        h = torch.view_as_complex((h1 + h2).reshape(nrhs, k, 2))
        assert (h - c[:, 0]).abs().max() < 64 * unit
        v = w / norm[:, None].to(rt)
    v = v.reshape(nrhs, n).to(torch.complex128)
    assert torch.einsum("krn,rn->kr", V[:k].to(torch.complex128).conj(), v).abs().max() < 16 * unit
    assert (v - Q[:, k]).abs().square().sum(1).max().sqrt() < 1e3 * 16 * unit
