"""What surrounds the FP64 fixed-point sweep (blocks above 16 MB of a grid
stencil).  A staged copy whose bounded wait gives up ends the solve with
LOGDET_ETIMEOUT, whichever of its products met it, and the next solve on the
same handle is exact; the memory estimate covers the values it keeps."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402

def _same(a, b):
    assert a.logdet == b.logdet and np.array_equal(a.per_probe, b.per_probe)


@pytest.mark.parametrize("method,k", [("oslq", 0), ("osaiop", 2)])
def test_wait_timeout_in_every_product(monkeypatch, method, k):
    # Every product of the solve stalls (20 ms a wait): the sketch product and
    # each step of OSLQ, both phases of OSA-IOP.
    with B.Handle.from_csr(W.laplacian_3d(52, 51, 50, shift=0.05)) as h:
        run = (lambda: h.oslq(60, 2, seed=1)) if method == "oslq" else \
            (lambda: h.osaiop(60, 2, iop_window=k, seed=1))
        want = run()
        monkeypatch.setenv("LOGDET_TEST_SWEEP_STALL", "1")
        with pytest.raises(B.LogdetError) as e:
            run()
        assert e.value.code == B.ETIMEOUT
        monkeypatch.delenv("LOGDET_TEST_SWEEP_STALL")
        _same(run(), want)


def test_wait_timeout_in_the_sketch_product_alone(monkeypatch):
    # LOGDET_TEST_SWEEP_STALL=sketch stalls the sketch product only: its Krylov
    # run waits for nothing that fails, so the product's own flag must report it.
    with B.Handle.from_csr(W.laplacian_3d(52, 51, 50, shift=0.05)) as h:
        want = h.oslq(60, 4, seed=1)
        monkeypatch.setenv("LOGDET_TEST_SWEEP_STALL", "sketch")
        with pytest.raises(B.LogdetError) as e:
            h.oslq(60, 4, seed=1)
        monkeypatch.delenv("LOGDET_TEST_SWEEP_STALL")
        assert e.value.code == B.ETIMEOUT
        _same(h.oslq(60, 4, seed=1), want)


def test_memory_estimate_counts_fixed_point_values():
    # The fixed-point values lie per row and diagonal, also where most rows have
    # no entry on a diagonal: 15 diagonals here, of which 12 hold one entry in 16.
    n, L = 300007, 500
    rows = np.arange(n)
    offs = [o for d in (1, 2, L - 1, L, L + 1, 2 * L, 3 * L) for o in (d, -d)]
    cols, vals, ptr = [rows], [np.full(n, 30.0)], [rows]
    for o in offs:
        lo = np.minimum(rows, rows + o)   # (the pair's smaller row decides, so that Q is symmetric)
        keep = (rows + o >= 0) & (rows + o < n) & ((abs(o) == 1) | (lo % 16 == 3))
        cols.append((rows + o)[keep])
        ptr.append(rows[keep])
        vals.append(np.full(keep.sum(), -1.0))
    r, c, v = (np.concatenate(x) for x in (ptr, cols, vals))
    order = np.lexsort((c, r))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    A = W.CSR(n, rowptr, c[order].astype(np.int32), v[order])
    nnz = len(v)
    dev = [torch.as_tensor(x, device="cuda") for x in (A.rowptr, A.colind, A.vals)]
    with B.Handle.from_csr(A) as hs, B.Handle(n, *dev, device=True) as hc:
        for probes, entries in ((24, 15 * n - nnz), (12, 0)):  # (a block below 16 MB: CSR values)
            a, b = (h.estimate_bytes(B.METHOD_OSLQ, probes, 8) for h in (hs, hc))
            assert a - b == 8 * entries
        x, y = (h.oslq(24, 8, seed=1) for h in (hs, hc))
        assert abs(x.logdet - y.logdet) <= 1e-12 * abs(y.logdet)
