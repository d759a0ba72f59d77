"""Matrices with a small leading block beside a large third diagonal entry,
against the oracle: the block (nearly) trace-free and the couplings to the
third axis along or near one of its eigenvectors, so that one spike and both
eigenvalues of the block are small at once -- FP32 lengths of eigenvectors
then come near underflow, where an FP32 frame once came out NaN and an
all-zero eigenvector matrix was taken for a solution."""

import numpy as np
import pytest

import oracle
import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1806_06698_gb300 import inputs  # noqa: E402

PERMS = [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]


@pytest.fixture(scope="module")
def syev3():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1806_06698_gb300 import build, syev3 as mod

    build.build()
    return mod


def packed(*entries):
    return np.stack(np.broadcast_arrays(*entries), axis=1).astype(np.float64)


def integer_blocks(rng, n, k):
    """a11 = -a22 = p, a12 = q with p = m^2 - j^2, q = 2 m j: the block's
    eigenvectors are (m, j) and (j, -m), which the couplings follow; the block
    2^-k of a33 = +-1."""
    m, j = rng.integers(1, 12, (2, n)).astype(np.float64)
    s, t, other = 2.0 ** -k / 128.0, rng.choice([-1.0, 1.0], n), rng.random(n) < 0.5
    p = m * m - j * j
    return packed(p * s, -p * s, t, 2.0 * m * j * s, np.where(other, j, m) * s, np.where(other, -m, j) * s)


def equal_couplings(rng, n, kind):
    """[[0, q, r], [q, 0, +-r], [r, +-r, 1]]."""
    u = rng.uniform(0.5, 1.5, (2, n))
    q, r = {
        "both": (1e-5 * u[0], 1e-5 * u[1]),
        "block": (4e-6 * u[0], 1e-3 * rng.standard_normal(n)),
        "spike": (1e-3 * rng.standard_normal(n), 1e-6 * u[1]),
        "larger": (3e-4 * u[0], 3e-4 * u[1]),
    }[kind]
    return packed(0.0 * q, 0.0 * q, 1.0, q, r, r * rng.choice([-1.0, 1.0], n))


def every_axis_order(A, rng):
    M = inputs.unpack(A) * rng.choice([-1.0, 1.0], (len(A), 1, 1)) * 2.0 ** rng.integers(-9, 10, (len(A), 1, 1))
    return np.concatenate([inputs.pack(M[i::6][:, p][:, :, p]) for i, p in enumerate(PERMS)])


def batch(kind, n=120000):
    rng = np.random.default_rng(2200 + sum(map(ord, kind)))
    if kind.startswith("integers"):
        return every_axis_order(integer_blocks(rng, n, int(kind.split("-")[1])), rng)
    return every_axis_order(equal_couplings(rng, n, kind), rng)


KINDS = ["both", "block", "spike", "larger"] + [f"integers-{k}" for k in (1, 4, 7, 8, 9, 10, 12)]


@pytest.mark.parametrize("kind", KINDS)
def test_fp64(syev3, kind):
    A = batch(kind)
    lam, U = syev3.syev3_batched(torch.from_numpy(A).cuda())
    lam_v, _ = syev3.syev3_batched(torch.from_numpy(A).cuda(), vectors=False)
    lam, U = lam.cpu().numpy(), U.cpu().numpy()
    parity.compare_f64(A, lam, U, *oracle.syev3(A))
    assert np.array_equal(lam_v.cpu().numpy(), lam)


@pytest.mark.parametrize("workspace", [False, True])
@pytest.mark.parametrize("kind", KINDS)
def test_compensated_fp32(syev3, kind, workspace):
    A = batch(kind).astype(np.float32)
    if workspace:  # above the size from which the workspace form refines from a list
        A = np.tile(A, ((1 << 21) // len(A) + 1, 1))
    At = torch.from_numpy(A).cuda()
    ws = torch.empty(syev3.workspace_bytes(len(A), At.dtype, compensated=True), dtype=torch.uint8, device="cuda")
    ctr = torch.zeros(syev3.NUM_COUNTERS, dtype=torch.int64, device="cuda")
    lam, U = syev3.syev3_batched(At, compensated=True, workspace=ws if workspace else None, counters=ctr)
    lam, U = lam.cpu().numpy(), U.cpu().numpy()
    m = len(batch(kind))
    parity.compare_f32(A[:m], lam[:m], U[:m], *oracle.syev3(A[:m].astype(np.float64)))
    if workspace:
        for lo in range(m, len(A), m):
            k = min(m, len(A) - lo)
            assert np.array_equal(lam[lo:lo + k], lam[:k]) and np.array_equal(U[lo:lo + k], U[:k])
    assert ctr[3].item() == 0


def test_integers(syev3):
    """One matrix that came back as (0, 0, 2^22) with zero eigenvectors."""
    A = np.array([[5.0, -5.0, -4194304.0, 12.0, 4.0, -6.0]])
    lam, U = syev3.syev3_batched(torch.from_numpy(A).cuda())
    parity.compare_f64(A, lam.cpu().numpy(), U.cpu().numpy(), *oracle.syev3(A))
    assert np.allclose(lam.cpu().numpy(), [[-4194304.0, -13.0, 13.0]], rtol=1e-4)
