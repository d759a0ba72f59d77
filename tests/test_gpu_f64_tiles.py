"""The FP64 solve with tiles of 64 matrices, for batches whose tiles are all
resident at once, and of 256: one result per matrix on both sides of the size
rule and at the edges of tiles, with few, many and only matrices left to the
FP64 path."""

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


def matrices(kind, n):
    if kind == "mixed":
        return inputs.mixed(n, seed=2600)[0]
    A = inputs.gaussian(n, seed=2601)
    if kind == "tridiagonal":
        A[:, 4] = 0.0
    return A


@pytest.mark.parametrize("kind", ["gaussian", "mixed", "tridiagonal"])
@pytest.mark.parametrize("offset", [0, 1])
def test_one_result_in_either_tile(syev3, kind, offset):
    """A batch past the rule in pieces of every remainder of a small tile."""
    line = torch.cuda.get_device_properties(0).multi_processor_count * 512
    A = matrices(kind, line + 300)
    buf = torch.zeros(A.size + 1, dtype=torch.float64, device="cuda")
    big = buf[offset:offset + A.size].view(-1, 6)
    big.copy_(torch.from_numpy(A))
    lam, U = syev3.syev3_batched(big)
    lam_v, _ = syev3.syev3_batched(big, vectors=False)
    assert torch.equal(lam, lam_v)
    cuts = [0, 1, 64, 127, 255, 512, 3000, 20001, 20001 + 63 * 64]
    for lo, hi in list(zip(cuts, cuts[1:])) + [(0, line), (0, line + 1)]:
        piece = big[lo:hi]
        for vectors in (True, False):
            lam_p, U_p = syev3.syev3_batched(piece, vectors=vectors)
            assert torch.equal(lam_p, lam[lo:hi])
            assert U_p is None or torch.equal(U_p, U[lo:hi])
    m = 20000
    parity.compare_f64(A[-m:], lam[-m:].cpu().numpy(), U[-m:].cpu().numpy(), *oracle.syev3(A[-m:]))
