"""Import and export of caller's arrays (axial frame rotation included) over every tile shape of the
line layout -- 1 to 8 sites per lane, short and padded lines, lattices of fewer lines than a tile,
one and several sources -- and over magnitudes on both sides of the range the exact-product FP32
rotation takes (2^-80 to 2^100), against the FP64 oracle. Tolerances: 1e-12 for FP64 steps; for FP32
steps 1e-6, about eight roundings of 2^-24 with a norm of M over its smallest output of order one."""

import numpy as np
import pytest

import synthetic as S
from oracle import wilson as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

# L, T: lanes per line and sites per lane differ in each (T = 5: padded, 37: 3 per lane, 160-256: long lines)
LATTICES = [(2, 2), (2, 5), (6, 16), (4, 27), (2, 37), (4, 64), (2, 120), (2, 160), (2, 190), (2, 250)]


@pytest.fixture(scope="module", params=[(c, ax) for c in LATTICES for ax in (True, False)],
                ids=lambda ca: f"L{ca[0][0]}T{ca[0][1]}-{'axial' if ca[1] else 'general'}")
def case(request):
    (L, T), axial = request.param
    p = W.Params(L, T, 0.065, xi=3.5, bc=-1)
    U = S.random_gauge(L, T, 0.3, 31)
    eta = S.gaussian_source(L, T, 131, nrhs=3)
    w = wf.Wilson(L, T, 0.065, kappa_t=3.5 * 0.065, bc=-1, axial=axial)
    w.load_gauge(U)
    yield p, U, eta, w
    w.close()


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("nrhs", [1, 3])
def test_full_fields(case, nrhs):
    p, U, eta, w = case
    x = torch.from_numpy(eta[:nrhs].copy()).cuda()
    for dagger, ref in ((False, W.M), (True, W.M_dag)):
        want = ref(U, eta[:nrhs], p)
        assert _rel(w.apply_M(x, dagger=dagger).cpu().numpy(), want) < 1e-12
        assert _rel(w.apply_M(x, dagger=dagger, f32=True).cpu().numpy(), want) < 1e-6


def test_magnitudes(case):
    """Sources scaled by powers of two: inside the exact-product range, outside it, and mixed with zeros."""
    p, U, eta, w = case
    want = W.M(U, eta, p)
    for k in ((0, -85, 60), (-75, 0, 95), (-95, 102, -60)):
        s = np.exp2(np.array(k, dtype=np.float64))
        x = eta * s.reshape((3,) + (1,) * (eta.ndim - 1))
        got = w.apply_M(torch.from_numpy(x).cuda(), f32=True).cpu().numpy()
        for i in range(3):
            assert _rel(got[i] / s[i], want[i]) < 1e-6, k
    point = np.zeros_like(eta)
    point[1].reshape(-1)[7] = 1.0
    got = w.apply_M(torch.from_numpy(point).cuda(), f32=True).cpu().numpy()
    assert _rel(got, W.M(U, point, p)) < 1e-6 and not got[0].any() and not got[2].any()


def test_not_finite(case):
    """A NaN or Inf stays in its own source and reaches the output there."""
    p, U, eta, w = case
    x = eta.copy()
    x[1].reshape(-1)[11] = np.nan
    x[2].reshape(-1)[3] = np.inf
    got = w.apply_M(torch.from_numpy(x).cuda(), f32=True).cpu().numpy()
    assert _rel(got[0], W.M(U, eta[0], p)) < 1e-6
    assert not np.isfinite(got[1]).all() and not np.isfinite(got[2]).all()
