"""Eigenvalues leave in ascending order, also where two of them differ only by
the solver's own rounding: rank-one and rank-two matrices, exact and rounded,
reflections and matrices of small integers, in every form."""

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


def batch(kind, n=60000):
    rng = np.random.default_rng(2300 + sum(map(ord, kind)))
    v, w = rng.standard_normal((2, n, 3))
    if kind == "integers":
        return rng.integers(-3, 4, (n, 6)).astype(np.float64)
    if kind == "integer vectors":
        v = rng.integers(-5, 6, (n, 3)).astype(np.float64)
    if kind == "reflections":
        v /= np.linalg.norm(v, axis=1)[:, None]
        return inputs.pack(np.eye(3) - 2.0 * v[:, :, None] * v[:, None, :])
    M = v[:, :, None] * v[:, None, :]
    if kind == "rank two":
        M = M + w[:, :, None] * w[:, None, :]
    return inputs.pack(M) * (-1.0 if kind == "negative" else 1.0)


@pytest.mark.parametrize("kind", ["rank one", "negative", "rank two", "integer vectors", "integers", "reflections"])
@pytest.mark.parametrize("form", ["fp64", "fp32", "compensated"])
def test_ascending(syev3, kind, form):
    A = batch(kind).astype(np.float64 if form == "fp64" else np.float32)
    At = torch.from_numpy(A).cuda()
    lam, U = syev3.syev3_batched(At, compensated=form == "compensated")
    lam_v, _ = syev3.syev3_batched(At, compensated=form == "compensated", vectors=False)
    lam, U = lam.cpu().numpy(), U.cpu().numpy()
    assert np.all(lam[:, :-1] <= lam[:, 1:])
    assert np.array_equal(lam_v.cpu().numpy(), lam)
    compare = parity.compare_f64 if form == "fp64" else parity.compare_f32
    compare(A, lam, U, *oracle.syev3(A.astype(np.float64)))
