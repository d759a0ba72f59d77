"""The compensated FP32 form where its refinement can go wrong, against the
oracle at the FP32 bar: every matrix flagged (a CTA's list runs full before
its last tile), tile edges, matrices outside the fixed-point refinement, and
the workspace form on both sides of its size rule, aligned and not; one
result per matrix whichever form solves it."""

import numpy as np
import pytest

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


def reflections(n, seed):
    """I - 2 v v^T scaled by 10^U(-6, 6): a double eigenvalue, always flagged."""
    rng = np.random.default_rng(seed)
    v = rng.standard_normal((n, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    M = (np.eye(3) - 2.0 * v[:, :, None] * v[:, None, :]) * 10.0 ** rng.uniform(-6.0, 6.0, (n, 1, 1))
    return inputs.pack(M).astype(np.float32)


def solve(mod, A, counters=None, workspace=False):
    At = A if isinstance(A, torch.Tensor) else torch.from_numpy(np.ascontiguousarray(A)).cuda()
    ws = None
    if workspace:
        ws = torch.empty(mod.workspace_bytes(len(At), At.dtype, compensated=True), dtype=torch.uint8, device="cuda")
    lam, U = mod.syev3_batched(At, compensated=True, counters=counters, workspace=ws)
    torch.cuda.synchronize()
    return lam, U


def check(A, lam, U):
    lam, U = lam.cpu().numpy(), U.cpu().numpy()
    lam_o, U_o = parity.oracle_all_cores(A.astype(np.float64))

    def part(lo, hi):
        sl = slice(lo, hi)
        parity.compare_f32(A[sl], lam[sl], U[sl], lam_o[sl], U_o[sl])

    parity.chunked(part, len(A), chunk=1 << 17)


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 1000, 1 << 20])
def test_all_flagged(syev3, n):
    A = reflections(n, 2100 + n)
    ctr = torch.zeros(syev3.NUM_COUNTERS, dtype=torch.int64, device="cuda")
    lam, U = solve(syev3, A, counters=ctr)
    check(A, lam, U)
    assert ctr[2].item() >= 0.9 * n and ctr[3].item() == 0


@pytest.mark.parametrize("log2", [-19, -21, -30])
def test_outside_the_fixed_point_range(syev3, log2):
    """Clustered 2x2 blocks with one coupling 2^log2 of the largest entry."""
    rng = np.random.default_rng(2120 - log2)
    n = 5000
    A = np.zeros((n, 6))
    t = rng.uniform(0.5, 1.0, n)
    A[:, 0] = t
    A[:, 1] = t * (1.0 + 1e-7 * rng.standard_normal(n))
    A[:, 2] = rng.uniform(-1.0, -0.5, n)
    A[:, 3] = 1e-7 * rng.standard_normal(n)
    A[:, 4] = 2.0 ** log2 * rng.standard_normal(n)
    A[:, 5] = 2.0 ** log2 * rng.standard_normal(n)
    A = A.astype(np.float32)
    check(A, *solve(syev3, A))


@pytest.mark.parametrize("n", [(1 << 21) - 1, (1 << 21) + 77])
@pytest.mark.parametrize("offset", [0, 1])
def test_workspace_form(syev3, n, offset):
    """Equal to the form without a workspace, bit for bit, counters included."""
    A = np.concatenate([inputs.mixed_fp32(1 << 18, seed=2130)[0], reflections(4096, 2131)])
    At = torch.from_numpy(A).cuda().repeat(n // len(A) + 2, 1)[offset:offset + n]
    c1 = torch.zeros(syev3.NUM_COUNTERS, dtype=torch.int64, device="cuda")
    c2 = torch.zeros_like(c1)
    lam1, U1 = solve(syev3, At, counters=c1)
    lam2, U2 = solve(syev3, At, counters=c2, workspace=True)
    assert torch.equal(c1, c2) and c1[2].item() > 0
    assert torch.equal(lam1, lam2) and torch.equal(U1, U2)
    m = len(A)
    check(np.roll(A, -offset, axis=0), lam1[:m], U1[:m])


@pytest.mark.parametrize("extra", [-1, 0, 1, 128, 255, 257])
def test_eigenvalues_only_in_long_tiles(syev3, extra):
    """The eigenvalues-only kernel on both sides of the size from which it
    takes longer tiles: those of the full solve, bit for bit."""
    n = (1 << 21) + extra
    A = torch.from_numpy(inputs.mixed_fp32(1 << 17, seed=2140)[0]).cuda().repeat(17, 1)[:n]
    lam_v, _ = syev3.syev3_batched(A)
    lam_n, U_n = syev3.syev3_batched(A, vectors=False)
    assert U_n is None and torch.equal(lam_v, lam_n)


@pytest.mark.parametrize("compensated", [False, True])
@pytest.mark.parametrize("decades", [2, 6, 12])
def test_spread_entries(syev3, decades, compensated):
    """Entries spread over many decades: starts far from the roots, so that
    lanes take the restart and the steps after the fixed schedule."""
    rng = np.random.default_rng(2150 + decades)
    A = (rng.standard_normal((1 << 17, 6)) * 10.0 ** rng.uniform(-decades, 0.0, (1 << 17, 6))).astype(np.float32)
    lam, U = syev3.syev3_batched(torch.from_numpy(A).cuda(), compensated=compensated)
    check(A, lam, U)


@pytest.mark.parametrize("base,vectors", [(1 << 19, False), (1 << 21, True)])
@pytest.mark.parametrize("extra", [-1, 0, 1, 129, 255])
def test_long_tiles_give_the_short_tiles_results(syev3, base, vectors, extra):
    """Both sides of the sizes from which a tile holds two matrices per thread:
    the results of the batch solved in short pieces, bit for bit."""
    n = base + extra
    A = torch.from_numpy(inputs.mixed_fp32(1 << 17, seed=2160)[0]).cuda().repeat(17, 1)[:n]
    lam, U = syev3.syev3_batched(A, vectors=vectors)
    for lo in range(0, n, 1 << 18):
        part = A[lo:lo + (1 << 18)].contiguous()
        lam_p, U_p = syev3.syev3_batched(part, vectors=vectors)
        assert torch.equal(lam[lo:lo + len(part)], lam_p)
        assert U is None or torch.equal(U[lo:lo + len(part)], U_p)
