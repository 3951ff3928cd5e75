"""Every transform length of the gridded operators, along each axis and in both
precisions, each shown to be the one that ran: quadratic forms of a Lanczos run
against a NumPy run on an FFT convolution (tolerances as in
test_gpu_gridfft.py: the FP64 bar 1e-10, the mixed budget 1e-4)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402
from test_gpu_gridfft import _convolve, _form  # noqa: E402


def _check(h, nx, ny, T, precision, probes=2, shift=0.25):
    G = O.rademacher_block(4, 1, nx * ny, probes)
    _, _, _, hi = h.info()
    r = h.oslq(probes, 2, seed=4, precision=precision, shift=shift, plain=1)
    c = hi + shift
    want = [_form(lambda v: (_convolve(v, nx, ny, T) + shift * v) / c, G[:, p], 2)
            for p in range(probes)]
    np.testing.assert_allclose(r.per_probe, want, rtol=1e-10 if precision == B.FP64 else 1e-4)


SHAPES = [(nx, ny, theta, precision, lengths)
          for precision in (B.FP64, B.MIXED_FP32)
          for nx, ny, theta, lengths in (
              (41, 43, 12.0, (6, 6)), (45, 40, 30.0, (7, 7)), (41, 40, 97.0, (8, 8)),
              (301, 40, 97.0, (9, 8)), (40, 303, 97.0, (8, 9)),
              (1401, 40, 97.0, (10, 8)), (40, 1403, 97.0, (8, 10)),     # two windows
              (1951, 121, 30.0, (11, 7)), (122, 1953, 30.0, (7, 11)),   # two windows
              (1201, 900, 50.0, None))]                                 # several windows each way


@pytest.mark.parametrize("nx,ny,theta,precision,lengths", SHAPES)
def test_length(nx, ny, theta, precision, lengths):
    T = W.wendland_table(theta, 0.5)
    with B.Handle.grid(nx, ny, T) as h:
        *got, windows = h.grid_transform(precision, 2)
        assert tuple(got) == lengths if lengths else windows > 2
        _check(h, nx, ny, T, precision)


def test_the_lengths_are_all_there():
    seen = {(p, axis, ln[axis]) for _, _, _, p, ln in SHAPES if ln for axis in (0, 1)}
    assert seen == {(p, axis, ln) for p in (B.FP64, B.MIXED_FP32) for axis in (0, 1)
                    for ln in range(6, 12)}


def test_direct_and_refused():
    with B.Handle.grid(64, 64, W.wendland_table(2.0, 0.5)) as h:
        assert h.grid_transform(B.FP64, 20) == (0, 0, 0)
        for precision, columns in ((B.MIXED_F32X2, 4), (B.FP64, 0)):
            with pytest.raises(B.LogdetError):
                h.grid_transform(precision, columns)
    with B.Handle.from_csr(W.laplacian_2d(8, 8, shift=1.0)) as h:
        with pytest.raises(B.LogdetError):
            h.grid_transform(B.FP64, 4)
