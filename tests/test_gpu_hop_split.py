"""FP64 fixed-point hops with the directions split over 6, 3, 2 warps and unsplit.

The number of sites in a call decides the split: a call with several sources and each source alone
run different ones. The sums are integers, exact but for the shifts to a common exponent (below a
quarter of an FP64 rounding of the largest term per direction): equal to 1e-14 of the result's norm,
for M, the preconditioned operator and the 4-D even-odd operator, in both frames, with padding slots,
and with neighbours whose exponents differ by up to 2^40.
"""

import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

# sites per 3-D parity / 32 of one source and of all: 36 -> 324; 128 -> 896; 256 -> 1280; 272 -> 1632
CASES = [(4, 33, 9), (8, 16, 7), (8, 32, 5), (8, 34, 6)]


@pytest.mark.parametrize("axial", [True, False], ids=["axial", "general"])
@pytest.mark.parametrize("L,T,nrhs", CASES)
def test_hop_split(L, T, nrhs, axial):
    w = wf.Wilson(L, T, 0.07, kappa_t=0.21, bc=-1, axial=axial)
    try:
        w.load_gauge(S.random_gauge(L, T, 0.3, 17 + T))
        x = torch.from_numpy(S.gaussian_source(L, T, 19 + T, nrhs=nrhs)).cuda()
        gen = torch.Generator(device="cuda").manual_seed(T)
        x = x * torch.exp2(torch.randint(-20, 21, x.shape[:-1], generator=gen, device="cuda").double()).unsqueeze(-1)
        xo = x.reshape(nrhs, -1, 12)[:, : L**3 * T // 2].reshape(nrhs, T, -1, 12).contiguous()
        ops = [(w.apply_M, x), (w.apply_schur, xo)] + ([(w.apply_eo4d, xo)] if T % 2 == 0 else [])
        for op, v in ops:
            for dagger in (False, True):
                many = op(v, dagger=dagger)
                for k in range(nrhs):
                    one = op(v[k : k + 1].contiguous(), dagger=dagger)
                    assert torch.linalg.norm(one[0] - many[k]) <= 1e-14 * torch.linalg.norm(many[k])
    finally:
        w.close()
