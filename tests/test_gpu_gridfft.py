"""Gridded operators applied by Fourier transforms (wide supports): every
transform length, one and several windows per axis, odd window counts, ragged
grids and column counts, against a NumPy Lanczos run on an FFT convolution.

m = 3 Lanczos steps exercise three applications per probe; the forms are held
to the FP64 bar (1e-10) and the mixed budget (1e-4)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402


def _convolve(x, nx, ny, T):
    R = T.shape[0] - 1
    my, mx = ny + 2 * R, nx + 2 * R   # room for every offset, also past the grid
    w = np.zeros((my, mx))
    d = np.arange(-R, R + 1)
    w[np.ix_(d % my, d % mx)] = T[np.ix_(abs(d), abs(d))]
    f = np.fft.rfft2(w)
    z = np.fft.rfft2(x.reshape(ny, nx), s=(my, mx))
    return np.fft.irfft2(z * f, s=(my, mx))[:ny, :nx].ravel()


def _form(apply, z, m):
    v, prev, beta = z / np.linalg.norm(z), 0.0, 0.0
    al, be = [], []
    for _ in range(m):
        w = apply(v)
        al.append(v @ w)
        w = w - al[-1] * v - beta * prev
        beta = np.linalg.norm(w)
        be.append(beta)
        prev, v = v, w / beta
    th, u = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
    return float((u[0] ** 2 * np.log(th)).sum())


@pytest.mark.parametrize("nx,ny,theta,probes", [
    (40, 43, 20.0, 3),       # one 64 x 64 window: no partner for it
    (64, 64, 33.0, 2),       # 128 points, grid as long as a power of two
    (301, 240, 20.0, 5),     # several windows along both axes
    (205, 97, 24.5, 3),
    (463, 464, 50.0, 2),     # n + R just at and past 512
    (1200, 90, 50.0, 4),     # long lines, short columns
    (70, 1500, 70.0, 2),     # the largest transforms along y
    (2500, 33, 30.0, 1),
    (33, 2500, 97.0, 1),     # radius 96
])
@pytest.mark.parametrize("precision,tol", [(B.FP64, 1e-10), (B.MIXED_FP32, 1e-4)])
def test_transformed_operator_forms(nx, ny, theta, probes, precision, tol):
    T = W.wendland_table(theta, 0.5)
    n, shift = nx * ny, 0.25
    G = O.rademacher_block(4, 1, n, probes)
    with B.Handle.grid(nx, ny, T) as h:
        _, _, _, hi = h.info()
        r = h.oslq(probes, 3, seed=4, precision=precision, shift=shift, plain=1)
    c = hi + shift
    want = [_form(lambda v: (_convolve(v, nx, ny, T) + shift * v) / c, G[:, p], 3)
            for p in range(probes)]
    np.testing.assert_allclose(r.per_probe, want, rtol=tol, atol=0)


def test_transformed_quadform_values_and_non_finite_fields():
    nx, ny = 301, 240
    T = W.wendland_table(30.0, 0.1)
    x = np.random.default_rng(1).standard_normal(nx * ny)
    want = float(x @ _convolve(x, nx, ny, T) + 0.5 * x @ x)
    with B.Handle.grid(nx, ny, T) as h:
        assert h.quadform(torch.as_tensor(x, device="cuda"), 0.5) == pytest.approx(want, rel=1e-12)
        for bad in (np.inf, np.nan):
            z = x.copy()
            z[77] = bad
            assert not np.isfinite(h.quadform(torch.as_tensor(z, device="cuda"), 0.5))


def test_transformed_operator_iop_server_and_plan():
    # OSA-IOP keeps its phase-1 basis (the last step has no free block to lend
    # as workspace); server and plan results equal the blocking call's bits.
    nx, ny = 231, 200
    with B.Handle.grid(nx, ny, W.wendland_table(25.0, 0.3)) as h:
        for precision in (B.FP64, B.MIXED_FP32):
            want = h.osaiop(15, 9, iop_window=3, seed=2, precision=precision)
            with B.Server(4 << 30) as srv:
                ids = [srv.submit(h, B.METHOD_OSAIOP, 15, 9, 3, seed=s, precision=precision)
                       for s in (1, 2)]
                got = [srv.wait(i) for i in ids][1]
            with B.Plan(h, B.METHOD_OSAIOP, 15, 9, 3, precision=precision) as plan:
                plan.run(7)
                again = plan.run(2)
            assert got.logdet == want.logdet == again.logdet
            assert np.array_equal(got.per_probe, want.per_probe)
            assert np.array_equal(again.per_probe, want.per_probe)
