"""The opt-in TMA-fed hop kernels (WF_TMA=1) of handles with lines of different length on threads of their own.

A launch's shared memory grows with the line; it must not depend on what another thread has just
launched. Results against the same handle's apply before the threads start, bit by bit.
"""

import threading

import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_0910_0992_gb300 as wf  # noqa: E402


def test_threads_of_different_lines(monkeypatch):
    monkeypatch.setenv("WF_TMA", "1")
    jobs = []
    for T in (32, 128, 32, 128):
        w = wf.Wilson(2, T, 0.07, kappa_t=0.24, bc=-1)
        stream = torch.cuda.Stream()
        w.set_stream(stream.cuda_stream)
        w.load_gauge(S.random_gauge(2, T, 0.3, T))
        x = torch.from_numpy(S.gaussian_source(2, T, T + 1)).cuda().reshape(-1, 12)[: 4 * T].reshape(1, T, 4, 12).contiguous()
        torch.cuda.synchronize()
        jobs.append((w, x, w.apply_schur(x, f32=True)))
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(jobs))

    def work(w, x, want):
        start.wait()
        try:
            for _ in range(500):
                got = w.apply_schur(x, f32=True)
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
