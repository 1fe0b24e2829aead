"""Full SW applies of several handles on host threads of their own, each lattice with another time extent.

The Q^-1 kernel's shared memory grows with the time extent and the number of sources; what one
thread's launch needs must not depend on what another thread has just launched. Results against the same
handle's apply before the threads start, bit by bit (one warp per line and source, no atomics).
"""

import threading

import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402

CASES = [(8, 1), (128, 4), (160, 4), (240, 3)]  # time extent, sources; L = 2


@pytest.mark.parametrize("f32", [True, False], ids=["fp32", "fp64"])
def test_threads_of_different_lattices(f32):
    jobs = []
    for T, nrhs in CASES:
        U = S.random_gauge(2, T, 0.3, T)
        w = wf.Wilson(2, T, 0.08, kappa_t=0.24, bc=-1)
        stream = torch.cuda.Stream()
        w.set_stream(stream.cuda_stream)
        w.load_gauge_clover(U, 1.1, 0.9)
        x = torch.from_numpy(S.gaussian_source(2, T, T + 1, nrhs=nrhs)).cuda()
        torch.cuda.synchronize()
        jobs.append((w, x, w.apply_Qinv(x, f32=f32)))
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(jobs))

    def work(w, x, want):
        start.wait()
        try:
            for _ in range(400):
                got = w.apply_Qinv(x, f32=f32)
            assert torch.equal(got, want)
        except Exception as e:  # reported below, in the test's own thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, _, _ in jobs:
        w.close()
    assert not errors, errors
