"""How exact the fixed-point products of the Hutch++ split are over all the
blocks they accept: columns whose largest entry is up to 16 times the mean, and
beyond, where the FP64 kernels take over.

An orthonormal column's squared norm differs from 1 by the error of the second
round's Gram entry (FP64 sums by tiles of 256 rows: 1.6e-16 to 2.9e-16 at these
sizes) and twice that of the reciprocal root (2 units, 2.2e-16): 1e-15 leaves
room for both.  The applies' roundings are independent over the rows and cancel.
Against the exact factor, in extended precision, a column is further off by the
rounding of its entries in two applies (1.1e-16 and less each): 4e-16 in the
2-norm."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_07004_gb300 import binding as B  # noqa: E402


def _block(n, s, rho, seed):
    """Gaussian columns with one entry just below a power of two, rho times the
    column's mean magnitude."""
    rng = np.random.default_rng(seed)
    y = rng.standard_normal((n, s))
    for c in range(s):
        f = 2.0 ** rng.integers(-6, 7)
        y[:, c] *= f / (rho * np.abs(y[:, c]).mean())
        assert np.abs(y[:, c]).max() < f
        y[rng.integers(n), c] = 0.99 * f
    return y


def _qr(y):
    y = y.astype(np.longdouble)
    c = np.einsum("ni,nj->ij", y, y)
    s = len(c)
    r = np.zeros_like(c)
    for j in range(s):
        r[j, j] = np.sqrt(c[j, j] - r[:j, j] @ r[:j, j])
        r[j, j + 1:] = (c[j, j + 1:] - r[:j, j] @ r[:j, j + 1:]) / r[j, j]
    a = np.empty_like(y)
    for j in range(s):
        a[:, j] = (y[:, j] - a[:, :j] @ r[:j, j]) / r[j, j]
    return a


@pytest.mark.parametrize("n,s", [(13007, 64), (20011, 32), (50021, 20), (400009, 7)])
@pytest.mark.parametrize("rho", [8.0, 15.5, 16.5, 31.0, 62.0])
def test_orthonormal_columns_over_the_accepted_range(n, s, rho):
    y = _block(n, s, rho, n + s)
    yd = torch.as_tensor(y, device="cuda")
    a = torch.empty_like(yd)
    assert B.logdet_orth(n, s, yd, s, a, s) == s
    a = a.cpu().numpy()
    norms = (a.astype(np.longdouble) ** 2).sum(0)
    off = float(np.abs(norms - 1).max())
    err = float(np.sqrt(((a - _qr(y)) ** 2).sum(0)).max())
    rms = float(np.sqrt(((a - _qr(y)) ** 2).sum(0).mean()))
    print(f"n {n} s {s} rho {rho}: norms {off:.1e}, columns {err:.1e} rms {rms:.1e}")
    assert off <= 1e-15
    assert err <= 4e-16


@pytest.mark.parametrize("n,s", [(50021, 20), (20011, 32)])
@pytest.mark.parametrize("kappa", [1e1, 1e3, 1e5])
def test_correlated_columns(n, s, kappa):
    # Columns of condition kappa, as a sketch's are: the applies' sums cancel, and
    # what an entry of Y or of the inverse factor loses counts kappa times.  The
    # FP64 kernels are off by 1.2e-17 to 3.1e-17 kappa there.
    rng = np.random.default_rng(7)
    u, v = (np.linalg.qr(rng.standard_normal((s, s)))[0] for _ in range(2))
    y = rng.standard_normal((n, s)) @ (u * np.logspace(0, -np.log10(kappa), s)) @ v
    yd = torch.as_tensor(y, device="cuda")
    a = torch.empty_like(yd)
    assert B.logdet_orth(n, s, yd, s, a, s) == s
    a = a.cpu().numpy()
    g = np.einsum("ni,nj->ij", a.astype(np.longdouble), a.astype(np.longdouble))
    assert np.abs(g - np.eye(s)).max() <= 1e-15
    assert np.sqrt(((a - _qr(y)) ** 2).sum(0)).max() <= 4e-16 + 3e-17 * kappa


@pytest.mark.parametrize("dtype,few,many", [
    # Where the FP64 (compensated FP32) kernels are faster, and where these are.
    (torch.float64, (4883, 64), (13007, 64)), (torch.float64, (9001, 50), (16001, 50)),
    (torch.float64, (40001, 20), (50021, 20)), (torch.float32, (400001, 50), (600001, 40)),
    (torch.float32, (300001, 24), (400001, 24))])
def test_which_products_a_block_takes(dtype, few, many):
    # The fixed-point products launch four kernels more a round (three for FP32).
    orth = B.logdet_orth if dtype == torch.float64 else B.logdet_orth_f32

    def launches(n, s):
        y = torch.randn(n, s, dtype=dtype, device="cuda")
        a = torch.empty_like(y)
        before = B.logdet_launch_count()
        orth(n, s, y, s, a, s)
        return B.logdet_launch_count() - before
    small = launches(1001, few[1])
    assert launches(*few) == small
    assert launches(*many) == small + (8 if dtype == torch.float64 else 6)
