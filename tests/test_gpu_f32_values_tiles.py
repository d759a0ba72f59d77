"""FP32 eigenvalues only, with one and with two matrices per thread and tile:
those of the full solve, bit for bit, on both sides of either kernel's size
rule (2^19 for eigenvalues only, 2^21 with eigenvectors)."""

import pytest

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


@pytest.mark.parametrize("base", [1 << 19, 1 << 21])
@pytest.mark.parametrize("extra", [-1, 0, 1, 255])
def test_values_of_the_full_solve(syev3, base, extra):
    n = base + extra
    A = torch.from_numpy(inputs.mixed_fp32(1 << 17, seed=2700)[0]).cuda().repeat(17, 1)[:n]
    lam, _ = syev3.syev3_batched(A)
    lam_v, U_v = syev3.syev3_batched(A, vectors=False)
    assert U_v is None and torch.equal(lam_v, lam)
