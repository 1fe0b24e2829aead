"""The FP64 hops in block fixed point against the FP64 oracle: sources whose exponents differ widely
between neighbouring sites and lines (the shared exponent then drops low bits of the small ones, an
error relative to the largest neighbour), sources near the ends of the served range, sites out of it
(the FP64 form), zeros and not-finite values. Tolerance 1e-14 relative to the result's norm: about
forty half-ulp roundings adding at random (0.3 x 2^-53 x sqrt(40)), times sixteen."""

import numpy as np
import pytest

import synthetic as S
from oracle import wilson as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

LATTICES = [(2, 2), (4, 6), (6, 16), (2, 37), (4, 48), (4, 128), (2, 160), (2, 250)]


@pytest.fixture(scope="module", params=[(c, ax) for c in LATTICES for ax in (True, False)],
                ids=lambda ca: f"L{ca[0][0]}T{ca[0][1]}-{'axial' if ca[1] else 'general'}")
def case(request):
    (L, T), axial = request.param
    p = W.Params(L, T, 0.065, xi=3.5, bc=-1)
    U = S.random_gauge(L, T, 0.4, 41)
    eta = S.gaussian_source(L, T, 141, nrhs=2)
    w = wf.Wilson(L, T, 0.065, kappa_t=3.5 * 0.065, bc=-1, axial=axial)
    w.load_gauge(U)
    yield p, U, eta, w
    w.close()


def _rel(a, b):
    m = np.abs(b).max()  # squares of these magnitudes would overflow or vanish
    a, b = a / m, b / m
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def _check(case, x, tol=1e-14):
    p, U, _, w = case
    for dagger, ref in ((False, W.M), (True, W.M_dag)):
        got = w.apply_M(torch.from_numpy(x).cuda(), dagger=dagger).cpu().numpy()
        want = ref(U, x, p)
        for k in range(x.shape[0]):
            assert _rel(got[k], want[k]) < tol, (k, dagger)


def test_exponents(case):
    """Gaussian, scaled per site by powers of two up to 2^+-200, and whole sources far up and down."""
    p, U, eta, w = case
    _check(case, eta)
    rng = np.random.default_rng(5)
    for span in (3, 40, 200):
        k = rng.integers(-span, span + 1, size=eta.shape[:5] + (1, 1))
        _check(case, eta * np.exp2(k.astype(np.float64)))
    _check(case, eta * np.exp2(np.array([-850.0, 900.0])).reshape(2, 1, 1, 1, 1, 1, 1))


def test_out_of_range(case):
    """Magnitudes the fixed-point form does not serve, alone and beside ordinary ones."""
    p, U, eta, w = case
    s = np.ones(eta.shape[:5] + (1, 1))
    s[0, 0, 0, 0, 0] = 2.0 ** 1010
    s[1] = 2.0 ** -950
    _check(case, eta * s)


def test_zero_and_not_finite(case):
    p, U, eta, w = case
    x = np.zeros_like(eta)
    x[1].reshape(-1)[5] = 1.0
    got = w.apply_M(torch.from_numpy(x).cuda()).cpu().numpy()
    assert not got[0].any() and _rel(got[1], W.M(U, x[1], p)) < 1e-14
    for bad in (np.nan, np.inf, -np.inf):
        x = eta.copy()
        x[1].reshape(-1)[17] = bad
        got = w.apply_M(torch.from_numpy(x).cuda()).cpu().numpy()
        assert _rel(got[0], W.M(U, eta[0], p)) < 1e-14
        # entry 17 is on the site x = 1, y = z = t = 0: that site and its spatial neighbours show it
        L = p.L
        for x_, y_, z_ in ((1, 0, 0), (2 % L, 0, 0), (0, 0, 0), (1, 1, 0), (1, L - 1, 0), (1, 0, 1), (1, 0, L - 1)):
            assert not np.isfinite(got[1, 0, z_, y_, x_]).all()
