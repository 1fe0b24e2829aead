"""The frame rotation of import and export, seen through what an operator leaves alone.

C_L returns spins 0 and 1, C_R spins 2 and 3 of its argument: import rotates them by g, export back by g^dag, nothing
else happens to them. On unit links g = 1 and the half comes back bit by bit. Links that are diagonal phases never
mix colours: each colour comes back within 256 x 2^-53 of itself, however far below the others it is (two
rotations, each with an error below 25 x 2^-53 of the colour in fixed point or 6 in FP64 arithmetic; the entries of g, products
of up to 15 phases whose moduli are off 1 by 1.5 x 2^-53 each and that round 4 times a product: 165). On
general links the error has no preferred sign: its mean over 98304 numbers of 4096 sites, in units of 2^-53 of the colour vector's norm,
is below 0.06 (errors of about 2 units that a site's g shares between its numbers: 2 / sqrt(24576) = 0.013 expected).
FP32: M-tilde_ILU without a clover term returns the even sites of its argument, rounded to FP32 in the frame. On
diagonal links each colour comes back within 2 x 2^-24 of itself: one rounding, and twice the split products' 0.48 x 2^-24
(174 x 2^-35 times the largest number of the vector, over 2^-6 of it at least, in each of the two parts).
"""

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

EPS = 2.0**-53


def _diagonal(L, T, phase):
    U = np.zeros((T, L, L, L, 4, 3, 3), dtype=np.complex128)
    a = np.random.default_rng(7).uniform(-np.pi, np.pi, U.shape[:5] + (2,)) * phase
    for k, v in enumerate((a[..., 0], a[..., 1], -a[..., 0] - a[..., 1])):
        U[..., k, k] = np.exp(1j * v)
    return U


def _gaussian(L, T, n, seed=3):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n, T, L, L, L, 4, 3)) + 1j * rng.standard_normal((n, T, L, L, L, 4, 3))


def _halves(U, psi):
    """The halves that C_L and C_R leave alone, put together: psi itself but for the rotations."""
    w = wf.Wilson(U.shape[1], U.shape[0], 0.065, kappa_t=3.5 * 0.065, bc=-1)
    try:
        w.load_gauge(U)
        x = torch.from_numpy(psi).cuda()
        return np.concatenate([w.apply_C(x, 0).cpu().numpy()[..., :2, :], w.apply_C(x, 1).cpu().numpy()[..., 2:, :]], -2)
    finally:
        w.close()


def _scaled(L, T):
    """Sources with colours 2^-30 apart, numbers scattered over 2^80, real and imaginary parts 2^-40 apart."""
    rng = np.random.default_rng(9)
    psi = _gaussian(L, T, 4)
    psi[0] *= np.array([1.0, 2.0**-30, 2.0**-60])
    psi[1] *= np.exp2(rng.uniform(-80, 0, psi[1].shape))
    psi[2] = psi[2].real + 1j * 2.0**-40 * psi[2].imag
    psi[3, ..., 1:] = 0.0
    return psi


@pytest.mark.parametrize("L,T", [(2, 5), (4, 16), (2, 160)])
def test_unit_links_exact(L, T):
    U = _diagonal(L, T, 0.0)
    for scale in (1.0, 2.0**-990, 2.0**900, 2.0**-1060):
        psi = _scaled(L, T) * scale
        assert np.array_equal(_halves(U, psi), psi)


def test_diagonal_links():
    L, T = 4, 16
    U = _diagonal(L, T, 1.0)
    for scale in (1.0, 2.0**-800, 2.0**900):
        psi = _scaled(L, T) * scale
        got = _halves(U, psi)
        assert (np.abs(got / scale - psi / scale) <= 256 * EPS * np.abs(psi / scale)).all()


def test_diagonal_links_fp32():
    L, T = 4, 16
    w = wf.Wilson(L, T, 0.065, kappa_t=3.5 * 0.065, bc=-1)
    try:
        w.load_gauge(_diagonal(L, T, 1.0))
        psi = _scaled(L, T)
        z, y, x = np.meshgrid(*[np.arange(L)] * 3, indexing="ij")
        even = (z + y + x) % 2 == 0
        got = w.apply_ilu(torch.from_numpy(psi).cuda(), f32=True).cpu().numpy()[:, :, even]
        want = psi[:, :, even]
        assert (np.abs(got - want) <= 2 * 2.0**-24 * np.abs(want)).all()
    finally:
        w.close()


def test_no_preferred_sign():
    L, T = 8, 8
    psi = _gaussian(L, T, 2)
    err = (_halves(S.random_gauge(L, T, 0.5, 4), psi) - psi) / np.linalg.norm(psi, axis=-1, keepdims=True) / EPS
    assert abs(err.real.mean()) < 0.06 and abs(err.imag.mean()) < 0.06


def test_not_finite():
    """A NaN or Inf reaches its own spin of its own site and nothing else."""
    L, T = 4, 16
    U = S.random_gauge(L, T, 0.5, 4)
    psi = _gaussian(L, T, 1)
    want = _halves(U, psi)
    for bad in (np.nan, np.inf, -np.inf):
        x = psi.copy()
        x[0, 5, 1, 2, 3, 0, 1] = bad
        ok = np.ones(x.shape, dtype=bool)
        ok[0, 5, 1, 2, 3, 0] = False
        got = _halves(U, x)
        assert np.array_equal(got[..., :2, :][ok[..., :2, :]], want[..., :2, :][ok[..., :2, :]])
        assert not np.isfinite(got[~ok]).any()
