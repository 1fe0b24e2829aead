"""FP64 hops component by component: a small spin or colour keeps FP64's accuracy beside a large one.

Each result component (spin and colour of a site) is held to a bound formed from its own terms alone: S,
the same operator with the absolute values of every factor, applied to |psi|. Fields whose spins, colours or
single components differ by up to 2^60, on links that do not mix colours (unity, diagonal phases), that
hardly do, and that do; one number of sites for each way the hop's directions are split over warps (6, 3, 2
and 1).

Tolerance 256 x 2^-53 S for one application of M: the fixed-point sums are used where their error is below
127 x 2^-53 S in each real number, 180 in a complex one (7.9 x 2^-53 times the largest number that enters
the result's spin, over a smallest S of 2^-4 of that); the hop's and the diagonal's remaining
operations and the oracle's own add below 20 roundings each, 28 in a complex number. Two hops (the 4-D
even-odd operator): twice that. In the axial frame the caller's colours are rotated (in FP64 arithmetic too),
so S is formed from colour norms there, at least the largest number itself: 16 x 2^-53 S from the sums, 28 as
above, and the rotations, the rotated links and their products below 200 roundings: 256 x 2^-53 S.
"""

import numpy as np
import pytest

import synthetic as S
from oracle import wilson as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

L, T = 4, 16
EPS = 2.0**-53
# sources: 512 sites of a 3-D parity each; 6 warps up to 9728 sites, 3 up to 24320, 2 up to 38912
SPLITS = [1, 24, 60, 80]


def _links(kind):
    if kind == "random":
        return S.random_gauge(L, T, 0.4, 5)
    if kind == "near unity":
        return S.random_gauge(L, T, 1e-4, 6)
    U = np.zeros((T, L, L, L, 4, 3, 3), dtype=np.complex128)
    a = np.random.default_rng(7).uniform(-np.pi, np.pi, U.shape[:5] + (2,)) * (kind == "diagonal")
    for k, v in enumerate((a[..., 0], a[..., 1], -a[..., 0] - a[..., 1])):
        U[..., k, k] = np.exp(1j * v)
    return U


def _fields(n, kinds=("spins", "far spins", "colours", "components", "one spin", "wide")):
    """n sources, of the kinds in turn."""
    rng = np.random.default_rng(11 + n)
    psi = rng.standard_normal((n, T, L, L, L, 4, 3)) + 1j * rng.standard_normal((n, T, L, L, L, 4, 3))
    for k in range(n):
        kind = kinds[k % len(kinds)]
        if kind.endswith("spins"):  # spins 0 and 3 meet in two axes and never meet 1 and 2 there
            f = 2.0**-20 if kind == "spins" else 2.0**-40  # (sums past 2^31 apart take the FP64 form)
            psi[k] *= np.array([f, 1.0, 1.0, f])[:, None]
            psi[k, :, :, :, 1::2] = 0.0  # along x only
        elif kind == "colours":
            psi[k] *= np.array([1.0, 2.0**-30, 2.0**-60])
        elif kind == "components":
            psi[k] *= np.exp2(rng.uniform(-12, 0, psi[k].shape))
        elif kind == "one spin":
            psi[k, ..., 1:, :] *= 2.0**-50
        else:
            psi[k] *= np.exp2(np.round(rng.uniform(-60, 0, psi[k].shape)))
    return psi


def _hops(U, x, p, norm):
    """S of D_t + D_s / gamma_f: absolute values throughout (norm: colour norms, links unitary)."""
    if norm:
        x, A = np.repeat(np.linalg.norm(x, axis=-1, keepdims=True), 3, -1), None
    out = 0.0
    for mu in range(4):
        f = 1.0 if mu == 3 else 1.0 / p.gamma_f
        A = np.abs(W.link(U, mu))
        fw, bw = W.shift(x, mu, 1, 1.0), W.shift(x, mu, -1, 1.0)
        if not norm:
            fw, bw = W.colour(A, fw), W.colour(W.dag(W.shift(A, mu, -1, 1.0)), bw)
        out = out + f * (W.spin(np.abs(W.I4 - W.GAMMA[mu]) / 2, fw) + W.spin(np.abs(W.I4 + W.GAMMA[mu]) / 2, bw))
    return out.real


def _worst(got, want, bound):
    err = np.abs(got - want)
    assert np.isfinite(err).all() and not err[bound == 0].any()
    return float((err[bound > 0] / bound[bound > 0]).max())


@pytest.fixture(scope="module", params=["unity", "diagonal", "near unity", "random"])
def lattice(request):
    return W.Params(L, T, 0.065, xi=3.5, bc=-1), _links(request.param)


@pytest.mark.parametrize("nrhs", SPLITS)
def test_M_components(lattice, nrhs):
    p, U = lattice
    w = wf.Wilson(L, T, 0.065, kappa_t=3.5 * 0.065, bc=-1, axial=False)
    try:
        w.load_gauge(U)
        psi = _fields(nrhs)
        for dagger, op in ((False, W.M), (True, W.M_dag)):
            size = np.roll(np.abs(psi), 2 * dagger, -2)  # |gamma_5|: spins s and s + 2 exchanged
            bound = np.roll(p.mu * size + _hops(U, size, p, False), 2 * dagger, -2)
            got = w.apply_M(torch.from_numpy(psi).cuda(), dagger=dagger).cpu().numpy()
            assert _worst(got, op(U, psi, p), bound) < 256 * EPS
    finally:
        w.close()


@pytest.mark.parametrize("nrhs", [1, 24])
def test_eo4d_components(lattice, nrhs):
    """mu - mu^-1 D^oe D^eo on the sites with x + y + z + t odd."""
    p, U = lattice
    w = wf.Wilson(L, T, 0.065, kappa_t=3.5 * 0.065, bc=-1, axial=False)
    try:
        w.load_gauge(U)
        t, z, y, x = np.meshgrid(*[np.arange(n) for n in (T, L, L, L)], indexing="ij")
        odd = ((t + z + y + x) % 2 == 1)
        psi = _fields(nrhs, ("colours", "components", "one spin", "wide")) * odd[..., None, None]

        def D(v):
            return W.D_t(U, v, p.bc) + W.D_s(U, v) / p.gamma_f

        want = p.mu * psi - D(D(psi)) / p.mu
        bound = p.mu * np.abs(psi) + _hops(U, _hops(U, np.abs(psi), p, False), p, False) / p.mu
        got = w.apply_eo4d(torch.from_numpy(psi[:, odd].copy()).cuda()).cpu().numpy()
        assert _worst(got, want[:, odd], bound[:, odd]) < 2 * 256 * EPS
    finally:
        w.close()


def test_axial_spins():
    """The axial frame mixes the colours of a spin, never spins."""
    p, U = W.Params(L, T, 0.065, xi=3.5, bc=-1), _links("random")
    w = wf.Wilson(L, T, 0.065, kappa_t=3.5 * 0.065, bc=-1)
    try:
        w.load_gauge(U)
        psi = _fields(6, ("spins", "far spins", "one spin"))
        norm = np.linalg.norm(psi, axis=-1, keepdims=True)
        bound = p.mu * np.repeat(norm, 3, -1) + _hops(U, psi, p, True)
        got = w.apply_M(torch.from_numpy(psi).cuda()).cpu().numpy()
        assert _worst(got, W.M(U, psi, p), bound) < 256 * EPS
    finally:
        w.close()
