"""FP64 line operations on both sides of the switch to one warp per spin.

A call with several sources of an 8^3 lattice has more than 608 lines and runs one warp per line;
each source alone has fewer and runs one warp per spin. The same arithmetic in the same order per
spin: equal to 1e-13 of the result's norm, in both frames, with and without padding slots, for T^-1
and the preconditioned operator (its hop in fixed point between them).
"""

import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402


@pytest.mark.parametrize("axial", [True, False], ids=["axial", "general"])
@pytest.mark.parametrize("T,nrhs", [(8, 10), (33, 3), (128, 3)])
def test_line_spin_matches_line(T, nrhs, axial):
    L = 8
    w = wf.Wilson(L, T, 0.07, kappa_t=0.21, bc=-1, axial=axial)
    try:
        w.load_gauge(S.random_gauge(L, T, 0.3, 7 + T))
        x = torch.from_numpy(S.gaussian_source(L, T, 9 + T, nrhs=nrhs)).cuda()
        xo = x.reshape(nrhs, T, -1, 12)[:, :, : L**3 // 2].contiguous()
        for op, v in ((lambda y, d: w.apply_Tinv(y, dagger=d), x), (lambda y, d: w.apply_schur(y, dagger=d), xo)):
            for dagger in (False, True):
                many = op(v, dagger)
                for k in range(nrhs):
                    one = op(v[k : k + 1].contiguous(), dagger)
                    assert torch.linalg.norm(one[0] - many[k]) <= 1e-13 * torch.linalg.norm(many[k])
    finally:
        w.close()
