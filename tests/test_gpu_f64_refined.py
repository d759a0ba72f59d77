"""The FP64 solve's two routes -- the FP32 solve refined in fixed point, for
matrices of similar entries, and the FP64 path for the rest -- against the
oracle at the FP64 bar, where each can go wrong: tile edges with the lists of
left-over matrices empty, partly full and full, entries at the border between
the routes, clusters of every width, and one result per matrix whatever its
neighbours, alignment or outputs."""

import numpy as np
import pytest

import oracle
import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_06698_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def syev3():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06698_gb300 import build, syev3 as mod

    build.build()
    return mod


def solve(mod, A, vectors=True):
    lam, U = mod.syev3_batched(torch.from_numpy(np.ascontiguousarray(A)).cuda(), vectors=vectors)
    torch.cuda.synchronize()
    return lam.cpu().numpy(), (U.cpu().numpy() if vectors else None)


def check(mod, A):
    lam, U = solve(mod, A)
    parity.compare_f64(A, lam, U, *oracle.syev3(A))
    return lam, U


def graded(A, rng, share):
    """A share of the matrices with one off-diagonal entry far below the rest."""
    A = A.copy()
    rows = rng.random(len(A)) < share
    A[rows, 3 + rng.integers(0, 3, rows.sum())] *= 2.0 ** -30
    return A


@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 511, 513, 304 * 256 + 77])
def test_tiles_and_lists(syev3, n, share):
    rng = np.random.default_rng(1700 + n)
    A = graded(inputs.gaussian(n, seed=1701 + n), rng, share)
    lam, _ = check(syev3, A)
    assert np.array_equal(solve(syev3, A, vectors=False)[0], lam)


@pytest.mark.parametrize("k", [0, 7, 8, 9, 12, 19, 20, 21, 22, 30])
def test_entry_spread(syev3, k):
    """Each entry in turn 2^-k of the others' size."""
    rng = np.random.default_rng(1720 + k)
    A = rng.uniform(0.5, 1.0, (6 * 400, 6)) * rng.choice([-1.0, 1.0], (6 * 400, 6))
    A[np.arange(6 * 400), np.arange(6 * 400) % 6] *= 2.0 ** -k
    check(syev3, A)


@pytest.mark.parametrize("k", [0, 10, 20, 27, 30, 40, 48, 52, 56, 60])
def test_clusters(syev3, k):
    """Two eigenvalues 2^-k apart, and three within 2^-k/2 of one another."""
    rng = np.random.default_rng(1740 + k)
    n = 1000
    t = 2.0 ** -k * rng.uniform(0.5, 1.0, n)
    one = np.ones(n)
    pair = inputs.conj_diag(inputs.haar(rng, n), np.stack([one, one + t, -rng.uniform(0.2, 3.0, n)], 1))
    triple = inputs.conj_diag(inputs.haar(rng, n), np.stack([one, one + t, one + 2.0 ** (-k // 2)], 1))
    check(syev3, np.concatenate([pair, triple]))


def test_exact_multiplicities(syev3):
    """Reflections I - 2 v v^T (a double eigenvalue) and rank-one matrices."""
    rng = np.random.default_rng(1760)
    v = rng.standard_normal((3000, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    P = v[:, :, None] * v[:, None, :]
    check(syev3, inputs.pack(np.concatenate([np.eye(3) - 2.0 * P, P])))


def test_each_matrix_alone(syev3):
    """A matrix's result does not depend on its place: shuffled, in an
    unaligned buffer and scaled by a power of two, bit for bit."""
    rng = np.random.default_rng(1770)
    A = np.concatenate([graded(inputs.gaussian(3000, seed=1771), rng, 0.2), inputs.mixed(2000, seed=1772)[0]])
    lam, U = check(syev3, A)
    p = rng.permutation(len(A))
    lam_p, U_p = solve(syev3, A[p])
    assert np.array_equal(lam_p, lam[p]) and np.array_equal(U_p, U[p])
    lam_s, U_s = solve(syev3, np.ldexp(A[:3000], -700))
    assert np.array_equal(lam_s, np.ldexp(lam[:3000], -700)) and np.array_equal(U_s, U[:3000])
    buf = torch.zeros(A.size + 1, dtype=torch.float64, device="cuda")
    buf[1:] = torch.from_numpy(A.reshape(-1)).cuda()
    lam_u, U_u = syev3.syev3_batched(buf[1:].view(-1, 6))
    torch.cuda.synchronize()
    assert np.array_equal(lam_u.cpu().numpy(), lam) and np.array_equal(U_u.cpu().numpy(), U)


@pytest.mark.parametrize("k", [24, 26, 27, 28, 29, 30, 40, 60])
def test_weak_coupling(syev3, k):
    """Nearly diagonal matrices with every coupling 2^-k of the smallest gap,
    one of them or two of them zero in some, at the border of the route that
    takes them by perturbation."""
    rng = np.random.default_rng(1780 + k)
    n = 6000
    d = np.stack([np.zeros(n), rng.uniform(1.0, 2.0, n), rng.uniform(3.0, 2000.0, n)], 1)
    d = rng.permuted(d - rng.uniform(0.0, 3.0, (n, 1)), axis=1)
    A = np.concatenate([d, 2.0 ** -k * rng.uniform(0.5, 1.0, (n, 3)) * rng.choice([-1.0, 1.0], (n, 3))], 1)
    A[: n // 3, 3] = 0.0
    A[: n // 6, 5] = 0.0
    A *= 10.0 ** rng.uniform(-50.0, 50.0, (n, 1))
    lam, _ = check(syev3, A)
    assert np.array_equal(solve(syev3, A, vectors=False)[0], lam)
