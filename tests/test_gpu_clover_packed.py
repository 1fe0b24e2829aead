"""FP32 clover blocks (lower triangles) and the adjoint of M-tilde_ILU.

The FP32 operators on lattices with one padded slot group, an odd time extent, half time extents
that leave a partial warp, and lines longer than 128 slots, against ``oracle/clover.py`` with the
FP32 tolerance of the operator tests (1e-6), and M-tilde_ILU's adjoint through <x, M y> = <M^dag x, y>
in FP64 (both sides are sums of 12 V terms: 1e-12 of |x| |M y|).
"""

import numpy as np
import pytest

import synthetic as S
from oracle import clover as CL
from oracle import wilson as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402


@pytest.mark.parametrize("axial", [True, False], ids=["axial", "general"])
@pytest.mark.parametrize("L,T", [(2, 3), (2, 34), (4, 5), (2, 130)])
def test_ilu_fp32_and_adjoint(L, T, axial):
    p = W.Params(L, T, 0.08, xi=3.0, bc=-1)
    U = S.random_gauge(L, T, 0.3, 41 + T)
    Acl = CL.clover_term(U, 1.1, 0.7)
    eta = S.gaussian_source(L, T, 51 + T, nrhs=2)
    par3 = W.parity3(L, T)
    w = wf.Wilson(L, T, 0.08, kappa_t=0.24, bc=-1, axial=axial)
    try:
        w.load_gauge_clover(U, 1.1, 0.7)
        x = torch.from_numpy(np.ascontiguousarray(eta)).cuda()
        for dagger, ref in ((False, CL.M_ilu(U, Acl, eta, p, par3)), (True, CL.M_ilu_dag(U, Acl, eta, p, par3))):
            got = w.apply_ilu(x, dagger=dagger, f32=True).cpu().numpy()
            assert np.linalg.norm((got - ref).ravel()) < 1e-6 * np.linalg.norm(ref.ravel())
        a = x[:1].contiguous()
        b = x[1:].contiguous()
        Mb = w.apply_ilu(b)
        lhs = torch.vdot(a.flatten(), Mb.flatten())
        rhs = torch.vdot(w.apply_ilu(a, dagger=True).flatten(), b.flatten())
        assert abs(lhs - rhs) < 1e-12 * torch.linalg.norm(a) * torch.linalg.norm(Mb)
    finally:
        w.close()
