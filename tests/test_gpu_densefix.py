"""The fixed-point products of the Hutch++ split (blocks with
n s^2 >= 2e7, FP32 2e8):
orth against an extended-precision QR at the edges of its tiles and row chunks, blocks
that leave the fixed-point range (heavy rows, infinities), dropped columns,
strides, and the projection through whole solves against the oracle.

Two rounds of Cholesky QR of a block with condition below 10 leave A within a
few units of 2^-53 (1.1e-16) times s of the exact factor in the 2-norm of a
column, for which 2e-14 (s <= 64) leaves room; FP32 blocks as many units of
2^-24, 1e-5."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402


def _block(n, s, seed, dtype=torch.float64):
    g = torch.Generator().manual_seed(seed)
    y = torch.randint(0, 2, (n + 2, s), generator=g).double() * 2 - 1
    y = 0.6 * y[1:-1] - 0.2 * y[:-2] - 0.2 * y[2:] + 0.1 * torch.randn(n, s, generator=g).double()
    # Every column has an exponent of its own, within the factor 1e6 beyond which orth drops one.
    scale = 10.0 ** torch.linspace(-2, 2, s)
    return (y * scale).to(dtype)


def _qr(y):
    """Y R^-1 with R the Cholesky factor of Y^T Y, in extended precision."""
    y = y.double().numpy().astype(np.longdouble)
    c = np.einsum("ni,nj->ij", y, y)
    s = len(c)
    r = np.zeros_like(c)
    for j in range(s):
        r[j, j] = np.sqrt(c[j, j] - r[:j, j] @ r[:j, j])
        r[j, j + 1:] = (c[j, j + 1:] - r[:j, j] @ r[:j, j + 1:]) / r[j, j]
    a = np.empty_like(y)
    for j in range(s):
        a[:, j] = (y[:, j] - a[:, :j] @ r[:j, j]) / r[j, j]
    return a.astype(np.float64)


def _run(y, pad=0, in_place=False):
    n, s = y.shape
    yd = torch.zeros(n, s + pad, dtype=y.dtype)
    yd[:, :s] = y
    yd = yd.cuda()
    a = yd if in_place else torch.full_like(yd, 7.0)
    f = B.logdet_orth if y.dtype == torch.float64 else B.logdet_orth_f32
    rank = f(n, s, yd, s + pad, a, s + pad)
    if pad and not in_place:
        assert (a[:, s:] == 7.0).all()
    return rank, a[:, :s].cpu().double().numpy()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n,s,pad,in_place", [
    (4883, 64, 0, False), (5121, 63, 1, True), (33000, 25, 3, False), (50000, 20, 0, True),
    (55001, 20, 20, False), (200129, 10, 2, True), (408231, 7, 1, False), (2300003, 3, 0, False),
    (12289, 64, 0, False), (49001, 64, 2, True), (50401, 63, 1, False), (80003, 25, 0, True),
    (500009, 20, 20, False), (502001, 10, 2, True), (2000003, 10, 0, False), (1040001, 7, 0, True)])
def test_orth_matches_qr(n, s, pad, in_place, dtype):
    y = _block(n, s, n + s, dtype)
    rank, a = _run(y, pad, in_place)
    tol = 2e-14 if dtype == torch.float64 else 1e-5
    assert rank == s
    assert np.abs(a.T @ a - np.eye(s)).max() <= tol
    assert np.linalg.norm(a - _qr(y), axis=0).max() <= tol


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_orth_heavy_row_takes_the_general_products(dtype):
    y = _block(510013, 20, 3, dtype)
    y[31007] *= 9e2
    rank, a = _run(y)
    tol = 2e-14 if dtype == torch.float64 else 1e-5
    assert rank == 20
    assert np.linalg.norm(a - _qr(y), axis=0).max() <= tol


def test_orth_drops_a_dependent_and_a_zero_column():
    y = _block(130013, 20, 4)
    y[:, 7] = 0.5 * y[:, 2] - 3.0 * y[:, 5]
    y[:, 11] = 0.0
    rank, a = _run(y)
    keep = [c for c in range(20) if c not in (7, 11)]
    assert rank == 18 and not a[:, [7, 11]].any()
    assert np.linalg.norm(a[:, keep] - _qr(y[:, keep]), axis=0).max() <= 2e-14


def test_orth_infinite_entry_ends_as_in_small_blocks():
    def parts(n):
        y = _block(n, 20, 5)
        y[1234, 3] = float("inf")
        rank, a = _run(y)
        return rank, np.isfinite(a).all(axis=0).tolist()
    assert parts(130013) == parts(40013)  # (the smaller block is below the fixed-point sizes)


@pytest.mark.parametrize("probes,gaussian", [(60, 0), (61, 0), (60, 1)])
def test_split_in_solves_matches_oracle(probes, gaussian):
    A = W.laplacian_2d(401, 320, shift=0.5)
    Q = A.to_scipy()
    with B.Handle.from_csr(A) as h:
        got = h.oslq(probes, 6, seed=3, gaussian=gaussian)
        low = h.oslq(probes, 6, seed=3, gaussian=gaussian, precision=B.MIXED_FP32)
    want = O.oslq(Q, probes, 6, seed=3, gaussian=bool(gaussian))
    assert abs(got.logdet - want.logdet) <= 1e-12 * abs(want.logdet)
    assert abs(low.logdet - want.logdet) <= 1e-6 * abs(want.logdet)
