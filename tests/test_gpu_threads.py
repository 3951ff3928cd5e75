"""Several host threads with shapes of their own at once: the calls share the
kernels' process-wide launch attributes (a kernel's limit of dynamic shared
memory), and every result must be that of the same call alone, bit for bit."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402


def _together(jobs, rounds):
    """Each job (a callable) `rounds` times on a thread of its own; its results
    must not differ from the first one, taken alone."""
    want = [job() for job in jobs]
    errors = []
    start = threading.Barrier(len(jobs))

    def work(job, expect):
        try:
            start.wait()
            for _ in range(rounds):
                got = job()
                assert all(np.array_equal(a, b) for a, b in zip(got, expect))
        except Exception as e:  # noqa: BLE001 (reported by the test)
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in zip(jobs, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_orthogonalisations_of_different_widths():
    def job(n, s):
        y = torch.randn(n, s, dtype=torch.float64, generator=torch.Generator().manual_seed(s)).cuda()
        a = torch.empty_like(y)
        st = torch.cuda.Stream()
        torch.cuda.synchronize()

        def run():
            rank = B.logdet_orth(n, s, y, s, a, s, stream=st.cuda_stream)
            st.synchronize()
            return rank, a[::997].cpu().numpy()
        return run
    _together([job(5121, 63), job(55001, 20), job(408231, 7)], 300)


def test_sweeps_of_different_stencils():
    hs = [B.Handle.from_csr(A) for A in (W.laplacian_3d(61, 60, 59, shift=0.05),
                                         W.laplacian_3d(211, 190, 5, shift=0.05),
                                         W.matern_2d(401, 0.05), W.matern_2d(301, 0.05))]
    try:
        jobs = []
        for i, h in enumerate(hs):
            def run(h=h, i=i):
                r = h.oslq(60 - 3 * i, 6, seed=i)
                f = h.oslq(30 + 12 * i, 6, seed=i, precision=B.MIXED_FP32)
                return r.logdet, r.per_probe, f.logdet, f.per_probe
            jobs.append(run)
        _together(jobs, 40)
    finally:
        for h in hs:
            h.close()
