"""FP64 eigenpairs of graded matrices D S D -- D a diagonal of powers of two, S
well conditioned -- to relative accuracy: small eigenvalues to their own size
and eigenvectors to rounding, where errors measured against the largest entry
cannot show a loss.

S has diagonal entries in [0.45, 1.1], couplings of at most 0.1 and relative
gaps of at least 0.2 in its diagonal.  An entrywise relative error of c eps in
A then moves an eigenvalue by at most c eps / (1 - 2 * 0.1 / 0.45) < 2 c eps of
itself and an eigenvector by that over the relative gap (at least 0.1 with the
couplings): with c = 8, the FP64 bar, 16 and 160 eps.
"""

import numpy as np
import pytest

import oracle
import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52
N = 20000


@pytest.fixture(scope="module")
def syev3():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06698_gb300 import build, syev3 as mod

    build.build()
    return mod


def graded(kind, k):
    """Exponents of D: every row but the first (or only the second) below it."""
    rng = np.random.default_rng(2400 + 64 * k + len(kind))
    S = np.empty((N, 6))
    S[:, :3] = np.array([1.0, 0.75, 0.5]) * rng.uniform(0.9, 1.1, (N, 3))
    S[:, 3:] = rng.uniform(0.05, 0.1, (N, 3)) * rng.choice([-1.0, 1.0], (N, 3))
    d = 2.0 ** -np.array({"two": [0, k, k], "one": [0, k, 0]}[kind])
    A = S * np.array([d[0] * d[0], d[1] * d[1], d[2] * d[2], d[0] * d[1], d[0] * d[2], d[1] * d[2]])
    if kind == "one":  # keep the gap of the two large ones
        A[:, 2] *= 0.5
    return A * 2.0 ** rng.integers(-300, 301, (N, 1))


def errors(A, lam, U):
    """Largest relative eigenvalue error and eigenvector error, in eps."""
    hi, lo, V = oracle.dd_jacobi(A)
    order = np.argsort(hi, axis=1)
    hi = np.take_along_axis(hi, order, 1)
    V = np.take_along_axis(V, order[:, None, :], 2)
    V = V * np.sign(np.sum(U * V, axis=1))[:, None, :]
    return np.max(np.abs(lam - hi) / np.abs(hi)) / EPS, np.max(np.linalg.norm(U - V, axis=1)) / EPS


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 14, 16])
@pytest.mark.parametrize("kind", ["two", "one"])
def test_relative_accuracy(syev3, kind, k):
    A = graded(kind, k)
    lam, U = syev3.syev3_batched(torch.from_numpy(A).cuda())
    lam_v, _ = syev3.syev3_batched(torch.from_numpy(A).cuda(), vectors=False)
    lam, U = lam.cpu().numpy(), U.cpu().numpy()
    assert np.array_equal(lam_v.cpu().numpy(), lam)
    assert np.all(lam[:, :-1] <= lam[:, 1:])
    parity.compare_f64(A, lam, U, *oracle.syev3(A))
    e_lam, e_vec = errors(A, lam, U)
    assert e_lam <= 16.0, f"eigenvalues off by {e_lam:.1f} eps of themselves"
    assert e_vec <= 160.0, f"eigenvectors off by {e_vec:.1f} eps"
