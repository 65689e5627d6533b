"""Rounding of the link update against extended precision.

U' = exp(i eps sum_a p_a lambda_a / 2) U with rows 0 and 1 orthonormalised, computed in the machine's
long double (64 or 113 bits) by a Taylor series of the 64th of Q, squared six times.  The rms error of the FP64
kernel must not exceed that of the language's square roots and divisions (9.3e-17 at eps = 0.1,
2.38e-16 at eps = 2, 3.44e-16 at eps = 3, measured with the kernel that used them) by more than the
scatter of 16,384 links' worth of entries (4 %).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD, CLD = np.longdouble, np.clongdouble


def _generators():
    T = np.zeros((8, 3, 3), CLD)
    h = LD(1) / 2
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        T[a, i, j] = T[a, j, i] = h
        T[a + 1, i, j], T[a + 1, j, i] = -1j * h, 1j * h
    T[2, 0, 0], T[2, 1, 1] = h, -h
    s3 = np.sqrt(LD(3))
    T[7, 0, 0] = T[7, 1, 1] = 1 / (2 * s3)
    T[7, 2, 2] = -1 / s3
    return T


def _mm(A, B):
    return (A[..., :, :, None] * B[..., None, :, :]).sum(-2)


def _expi(Q):
    A = Q * CLD(1j) / 64
    E = np.zeros_like(A)
    E[..., range(3), range(3)] = 1
    term = E.copy()
    for k in range(1, 26):
        term = _mm(term, A) / k
        E = E + term
    for _ in range(6):
        E = _mm(E, E)
    return E


def _rows(U):
    U = U.copy()
    U[..., 0, :] /= np.sqrt((np.abs(U[..., 0, :]) ** 2).sum(-1))[..., None]
    U[..., 1, :] -= (U[..., 0, :].conj() * U[..., 1, :]).sum(-1)[..., None] * U[..., 0, :]
    U[..., 1, :] /= np.sqrt((np.abs(U[..., 1, :]) ** 2).sum(-1))[..., None]
    U[..., 2, :] = np.cross(U[..., 0, :], U[..., 1, :]).conj()
    return U


@pytest.mark.skipif(np.finfo(LD).nmant <= 52, reason="long double is no wider than double")
def test_rms_error():
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    dims = (8, 8, 8, 8)
    lat = wd.Lattice(dims)
    V, T, rng = lat.V, _generators(), np.random.default_rng(11000)
    U0 = _rows(_expi(np.tensordot(rng.standard_normal((V, 4, 8)).astype(LD) / 2, T, axes=1))).astype(np.complex128)
    for eps, most in ((0.1, 9.3e-17), (2.0, 2.38e-16), (3.0, 3.44e-16)):
        p = rng.standard_normal((V, 4, 8))
        lat.wd_gauge_load(torch.from_numpy(U0.view(np.float64).reshape(-1)).cuda())
        P = lat.algebra_field()
        lat.wd_algebra_pack(torch.from_numpy(p.reshape(-1)).cuda(), P)
        lat.step_T(P, eps)
        out = torch.empty(72 * V, dtype=torch.float64, device="cuda")
        lat.wd_gauge_store(out)
        got = out.cpu().numpy().view(np.complex128).reshape(V, 4, 3, 3).astype(CLD)
        ref = _rows(_mm(_expi(np.tensordot(p.astype(LD) * LD(eps), T, axes=1)), U0.astype(CLD)))
        rms = float(np.sqrt((np.abs(got - ref) ** 2).mean()))
        print(eps, rms)
        assert rms < 1.04 * most, (eps, rms)
    lat.close()
