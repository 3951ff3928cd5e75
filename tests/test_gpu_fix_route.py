"""Which SpMM pass an FP64 solve takes: the fixed-point sweep counts as one
profiled pass like the CSR pass, and launches one kernel more a pass.  Every
matrix and window of the comparisons of the two passes is shown to take the
sweep from host arrays, and what must not take it to take the CSR pass."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402
import test_gpu_fix as F  # noqa: E402
import test_gpu_fix_range as R  # noqa: E402


def _counts(h, run):
    """(profiled SpMM passes, kernels launched) of one solve."""
    run(h)
    B.logdet_profile_reset()
    B.logdet_profile_enable(True)
    before = B.logdet_launch_count()
    run(h)
    launched = B.logdet_launch_count() - before
    B.logdet_profile_enable(False)
    passes = B.logdet_profile_read(0)["launches"]
    B.logdet_profile_reset()
    return passes, launched


MATRICES = {**F.MATRICES, **{"raised " + k: v for k, v in R.MATRICES.items()},
            "patch": lambda: F._patch(-1.0)}


@pytest.mark.parametrize("name", sorted(MATRICES))
@pytest.mark.parametrize("k", [0, 2, 4, 8])
def test_host_arrays_of_a_grid_stencil_take_the_sweep(name, k):
    run = (lambda h: h.osaiop(60, 6, iop_window=k, seed=3)) if k else (lambda h: h.oslq(60, 6, seed=3))
    fix, csr = F._both(MATRICES[name]())
    with fix, csr:
        (p1, l1), (p0, l0) = _counts(fix, run), _counts(csr, run)
    assert p1 == p0 == (12 if k else 7)
    # One kernel more a pass, and each step but the last its norm by itself.
    # The sweep's values take one kernel as the CSR values do.
    assert l1 - l0 == p1 + (10 if k else 5)


def test_small_unbalanced_and_grouped_solves_take_the_csr_pass():
    run = lambda h: h.oslq(60, 6, seed=3)  # noqa: E731
    A = W.laplacian_2d(409, 401, shift=0.5)
    heavy = W.laplacian_2d(409, 401, shift=0.5)
    row = 200 * 409 + 77
    q = heavy.rowptr[row] + int(np.flatnonzero(
        heavy.colind[heavy.rowptr[row]:heavy.rowptr[row + 1]] == row)[0])
    heavy.vals[q] = 4e6
    for M, r in ((heavy, run), (W.laplacian_2d(301, 300, shift=0.5), run),
                 (A, lambda h: h.oslq_shifts([0.0, 0.1], 30, 6, seed0=1))):
        fix, csr = F._both(M)
        with fix, csr:
            assert _counts(fix, r) == _counts(csr, r)
