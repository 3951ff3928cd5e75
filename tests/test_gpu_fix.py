"""The fixed-point SpMM sweep of FP64 blocks (grid stencils from host arrays,
blocks above 16 MB) against the CSR pass, which the same matrix takes when it
is handed over as device arrays: line and plane sweeps, every compiled
diagonal count and the general one, ragged grids and tiles, window widths,
shifts, slices, and vectors that leave the fixed-point range.

Both sides round differently at 2^-53; the estimators amplify that by well
under 1e3 on these matrices (the FP64 oracle moves by < 1e-15 between dot
orders), so the estimates are held to 1e-12 and the forms to 1e-11."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402


def _both(A):
    dev = [torch.as_tensor(x, device="cuda") for x in (A.rowptr, A.colind, A.vals)]
    torch.cuda.synchronize()
    return B.Handle.from_csr(A), B.Handle(A.n, *dev, device=True)


def _close(a, b, rtol=1e-12):
    assert abs(a.logdet - b.logdet) <= rtol * abs(b.logdet)
    np.testing.assert_allclose(a.per_probe, b.per_probe, rtol=10 * rtol, atol=10 * rtol)
    np.testing.assert_allclose(a.z_norm2, b.z_norm2, rtol=rtol)
    assert (a.steps_min, a.steps_max, a.status_bits) == (b.steps_min, b.steps_max, b.status_bits)


MATRICES = {
    "lap3d": lambda: W.laplacian_3d(59, 61, 47, shift=0.03),
    "lap3d_flat": lambda: W.laplacian_3d(211, 190, 5, shift=0.03),
    "lap2d": lambda: W.laplacian_2d(433, 397, shift=0.05),
    "matern": lambda: W.matern_2d(401, 0.05),
    "box3d": lambda: W.grid_stencil_3d(61, 53, 51, [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0),
                                                    (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
                                                    (0, 1, 1), (0, -1, -1)]),
    "lap3d_f32": lambda: W.laplacian_3d(57, 55, 53, shift=0.03, dtype=np.float32),
}


@pytest.mark.parametrize("name", sorted(MATRICES))
@pytest.mark.parametrize("method,k,probes", [("oslq", 0, 60), ("osaiop", 2, 63), ("osaiop", 4, 60),
                                             ("osaiop", 8, 60)])
def test_fixed_point_sweep_equals_csr_pass(name, method, k, probes):
    if method == "osaiop" and k > 2 and name not in ("lap3d", "matern"):
        pytest.skip("window widths are covered on two matrices")
    fix, csr = _both(MATRICES[name]())
    with fix, csr:
        if method == "oslq":
            kw = dict(shift=0.02, gaussian=1) if name == "lap2d" else {}
            _close(fix.oslq(probes, 14, seed=3, **kw), csr.oslq(probes, 14, seed=3, **kw))
        else:
            kw = dict(shift=0.4) if k == 2 else {}
            _close(fix.osaiop(probes, 12, iop_window=k, seed=3, **kw),
                   csr.osaiop(probes, 12, iop_window=k, seed=3, **kw))


def test_fixed_point_sweep_oracle_slices_server_and_plan():
    A = W.laplacian_3d(52, 51, 50, shift=0.05)
    est = O.oslq(A.to_scipy(), 60, 8, seed=1)
    with B.Handle.from_csr(A) as h:
        r = h.oslq(60, 8, seed=1)
        assert abs(r.logdet - est.logdet) <= 1e-10 * abs(est.logdet)
        np.testing.assert_allclose(r.per_probe, est.per_probe, rtol=1e-9, atol=1e-9)
        _close(h.oslq(60, 8, seed=1, block_width=20), r)
        with B.Server(8 << 30) as srv:
            ids = [srv.submit(h, B.METHOD_OSLQ, 60, 8, seed=s) for s in (0, 1)]
            ids.append(srv.submit(h, B.METHOD_OSAIOP, 60, 8, 4, seed=1))
            got = [srv.wait(i) for i in ids]
        assert got[1].logdet == r.logdet and np.array_equal(got[1].per_probe, r.per_probe)
        assert got[2].logdet == h.osaiop(60, 8, iop_window=4, seed=1).logdet
        with B.Plan(h, B.METHOD_OSLQ, 60, 8) as plan:
            assert plan.run(1).logdet == r.logdet


def _patch(value):
    # 5 I with a 5-point patch of couplings: after the first step a Lanczos
    # vector lives on the patch alone, hundreds of times its root mean square.
    A = W.laplacian_2d(409, 401, shift=1.0)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    x, y = rows % 409, rows // 409
    cx, cy = A.colind % 409, A.colind // 409
    inside = (abs(x - 200) < 6) & (abs(y - 200) < 6) & (abs(cx - 200) < 6) & (abs(cy - 200) < 6)
    off = A.colind != rows
    A.vals[off] = np.where(inside[off], value, 0.0)
    return A


@pytest.mark.parametrize("method", ["oslq", "osaiop"])
def test_vectors_outside_the_fixed_point_range(method):
    fix, csr = _both(_patch(-1.0))
    with fix, csr:
        run = (lambda h: h.oslq(60, 6, seed=2)) if method == "oslq" else \
            (lambda h: h.osaiop(60, 6, iop_window=2, seed=2))
        _close(run(fix), run(csr))


def test_unbalanced_rows_take_the_csr_pass():
    A = W.laplacian_2d(409, 401, shift=0.5)
    row = 200 * 409 + 77
    q = A.rowptr[row] + int(np.flatnonzero(A.colind[A.rowptr[row]:A.rowptr[row + 1]] == row)[0])
    A.vals[q] = 4e6
    fix, csr = _both(A)
    with fix, csr:
        a, b = (h.osaiop(60, 6, iop_window=2, seed=2) for h in (fix, csr))
    assert a.logdet == b.logdet and np.array_equal(a.per_probe, b.per_probe)
