"""The force's CG replayed as a CUDA graph (a handle with a stream of its own) against plain launches.

The same iteration, run as launches on the default stream and as graph replays on the handle's own,
and cut at an iteration limit inside a block. Both are solved to 1e-12, so force and action agree to
1e-10 of their size; the iteration counts are equal or one apart (the norms are sums of atomics).
"""

import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("L,T", [(2, 5), (4, 16), (4, 128)])
def test_force_graph_matches_launches(L, T, precision):
    U = S.random_gauge(L, T, 0.3, 61 + T)
    rng = np.random.default_rng(T)
    shape = (T, L**3 // 2, 12)
    phi = torch.from_numpy(rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).cuda()
    out = []
    for own in (False, True):
        stream = torch.cuda.Stream()
        w = wf.Wilson(L, T, 0.075, kappa_t=0.225, bc=-1)
        try:
            if own:
                w.set_stream(stream.cuda_stream)
            torch.cuda.synchronize()
            w.load_gauge(U)
            F = torch.empty(T, L, L, L, 4, 8, dtype=torch.float64, device="cuda")
            action, iters = wf.wf_force(w.h, phi, F, precision, 1e-12)
            torch.cuda.synchronize()
            out.append((action, iters, F))
            wf.wf_set_max_iterations(w.h, 3)
            assert wf.wf_force(w.h, phi, None, precision, 1e-12)[1] == 3
        finally:
            w.close()
    (s0, i0, f0), (s1, i1, f1) = out
    assert abs(i0 - i1) <= 1
    assert abs(s0 - s1) <= 1e-10 * abs(s0)
    assert torch.linalg.norm(f0 - f1) <= 1e-10 * torch.linalg.norm(f0)
