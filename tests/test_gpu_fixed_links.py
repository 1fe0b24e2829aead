"""The fixed-point links of the FP64 hops: formed when an FP64 operator first needs them, and FP64 arithmetic without them.

They take as much memory as the FP64 links; a handle that only makes FP32 applies does not hold
them. Environment WF_FX=0 stands for a device without room for them: every site then takes the general (FP64) form, and
agrees with the fixed-point form to 1e-14 of the result's norm (each is within 40 roundings of 2^-53 at random, and the
frame rotations around both are the same).
"""

import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

MB = 1 << 20


def test_fp32_handle_does_not_hold_them():
    L, T = 16, 64
    U = torch.from_numpy(S.random_gauge(L, T, 0.3, 1)).cuda()
    x = torch.from_numpy(S.gaussian_source(L, T, 2)).cuda().reshape(-1, 12)[: L**3 * T // 2].reshape(1, T, -1, 12).contiguous()
    warm = wf.Wilson(2, 64, 0.07, kappa_t=0.24, bc=-1)  # the kernels' code and torch's own buffers
    warm.load_gauge(S.random_gauge(2, 64, 0.3, 1))
    warm.apply_schur(x.reshape(-1)[: 4 * 64 * 12].reshape(1, 64, 4, 12).contiguous(), f32=True)
    w = wf.Wilson(L, T, 0.07, kappa_t=0.24, bc=-1)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    w.load_gauge(U)
    out = w.apply_schur(x, f32=True)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    V = L**3 * T
    links = V * (3 * 144 + 144 + 3 * 48)  # FP64 spatial and temporal links, FP32 two-row spatial links
    fields = 8 * V // 2 * 96 + 2 * out.numel() * 16
    assert used < links + fields + 32 * MB < links + fields + V * 432, used / MB
    w.close()
    warm.close()


@pytest.mark.parametrize("axial", [True, False], ids=["axial", "general"])
@pytest.mark.parametrize("L,T,nrhs", [(2, 5, 1), (4, 16, 2), (8, 32, 5), (4, 130, 3)])
def test_general_form_agrees(L, T, nrhs, axial, monkeypatch):
    U, U2 = S.random_gauge(L, T, 0.3, 7), S.random_gauge(L, T, 0.3, 8)
    x = torch.from_numpy(S.gaussian_source(L, T, 9, nrhs=nrhs)).cuda()
    xo = x.reshape(nrhs, -1, 12)[:, : L**3 * T // 2].reshape(nrhs, T, -1, 12).contiguous()
    w, g = (wf.Wilson(L, T, 0.07, kappa_t=0.21, bc=-1, axial=axial) for _ in range(2))
    try:
        for V in (U, U2):  # the second field replaces the first on handles that have used it
            w.load_gauge(V)
            monkeypatch.setenv("WF_FX", "0")
            g.load_gauge(V)
            for name, v in [("apply_M", x), ("apply_schur", xo)] + ([("apply_eo4d", xo)] if T % 2 == 0 else []):
                for dagger in (False, True):
                    monkeypatch.setenv("WF_FX", "0")
                    want = getattr(g, name)(v, dagger=dagger)
                    monkeypatch.delenv("WF_FX")
                    got = getattr(w, name)(v, dagger=dagger)
                    assert torch.linalg.norm(got - want) <= 1e-14 * torch.linalg.norm(want), (name, dagger)
                    assert not torch.equal(got, want), name  # two routes
        monkeypatch.setenv("WF_FX", "0")
        sol, _, res, status = g.solve(x, tol=1e-10)
        assert status == wf.WF_OK and max(res) <= 1e-10
    finally:
        w.close()
        g.close()
