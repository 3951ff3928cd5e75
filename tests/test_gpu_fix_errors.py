"""Wait failures of the FP64 fixed-point sweep (blocks above 16 MB of a grid
stencil): a staged copy whose bounded wait gives up ends the solve with
LOGDET_ETIMEOUT, whichever of its products met it, and the next solve on the
same handle is exact."""
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
