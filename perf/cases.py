"""The work that is timed: calls of the batched eigensolver's public entry
points, from one small batch to the largest ones, in both element types.

Inputs are built on the GPU as A = Q diag(z) Q^T with Q from a seeded unit
quaternion, so that a case's reference values follow from its construction.
The recipes are those of ``paper_1806_06698_gb300/inputs.py`` (well-separated
spectra, clustered spectra, near-diagonal and exactly diagonal matrices,
positive structure tensors) plus matrices with one principal axis in the
xy-plane (plane-strain-like tensors in a rotated frame), whose smaller arrow
spike is at rounding level.  Where eigenvectors are returned, spectra keep the
eigenvectors determined to the element type's accuracy and no eigenvector has
its two largest components nearly equal: there the sign rule has two correct
answers.
"""

import math

import torch

from paper_1806_06698_gb300 import syev3

CHUNK = 1 << 21  # matrices built at a time
FLOPS = 313.7    # floating-point operations of the method per matrix (mixed batch)
FLOPS_BWD = 138.0

# Shares of spectral, clustered, near-diagonal, exactly diagonal and plane
# matrices; log10 range of the clustered gap; log10 of the scale range; kind
# of spectrum; smallest relative gap.
RECIPES = {
    "mixed64": ((0.6, 0.2, 0.1, 0.1, 0.0), (2.0, 5.0), 50.0, "normal", 1e-3),
    "mixed64_values": ((0.6, 0.2, 0.1, 0.1, 0.0), (2.0, 14.0), 50.0, "normal", 1e-3),
    "mixed32": ((0.6, 0.2, 0.1, 0.1, 0.0), (1.0, 2.0), 6.0, "normal", 1e-2),
    "plane32": ((0.5, 0.0, 0.1, 0.1, 0.3), (1.0, 2.0), 6.0, "normal", 1e-2),
    "tensors": ((1.0, 0.0, 0.0, 0.0, 0.0), (1.0, 2.0), 3.0, "positive", 1e-2),
    "spectral": ((1.0, 0.0, 0.0, 0.0, 0.0), (1.0, 2.0), 0.0, "normal", 1e-2),
}


def listed():
    return [
        # The small parity workload: one call on 4096 matrices, where launch and host latency count.
        {"name": "solve_f64_small", "call": "solve", "dtype": "f64", "n": 4096, "recipe": "spectral", "vectors": True},
        # The headline workload: 2^24 mixed-difficulty FP64 matrices, eigenvalues and eigenvectors.
        {"name": "solve_f64_mixed", "call": "solve", "dtype": "f64", "n": 1 << 24, "recipe": "mixed64", "vectors": True},
        # Eigenvalues alone (invariants, stability checks) of an odd number of mixed FP64 matrices.
        {"name": "values_f64", "call": "solve", "dtype": "f64", "n": 1000003, "recipe": "mixed64_values",
         "vectors": False},
        # Structure tensors of a 67^3 volume in FP32.
        {"name": "solve_f32_tensors", "call": "solve", "dtype": "f32", "n": 67 ** 3, "recipe": "tensors",
         "vectors": True},
        # The FP32 headline workload: 2^24 mixed matrices.
        {"name": "solve_f32_mixed", "call": "solve", "dtype": "f32", "n": 1 << 24, "recipe": "mixed32", "vectors": True},
        # Eigenvalue filters (vesselness, cornerness) over a large volume: FP32 eigenvalues alone.
        {"name": "values_f32", "call": "solve", "dtype": "f32", "n": 323 ** 3, "recipe": "tensors", "vectors": False},
        # Compensated FP32, refinement inside the call, a ragged batch.
        {"name": "comp_f32", "call": "comp", "dtype": "f32", "n": 777777, "recipe": "plane32", "vectors": True},
        # Compensated FP32 with a caller's workspace, a large batch.
        {"name": "comp_ws_f32", "call": "comp_ws", "dtype": "f32", "n": 1 << 23, "recipe": "plane32", "vectors": True},
        # One training step's eigendecomposition in FP64: forward and backward through autograd.
        {"name": "train_f64", "call": "train", "dtype": "f64", "n": 131071, "recipe": "spectral"},
        # The backward kernel alone at the differentiation workload's size, FP32.
        {"name": "bwd_f32", "call": "bwd", "dtype": "f32", "n": 1 << 20, "recipe": "spectral"},
        # End to end from pinned host memory, FP64.
        {"name": "host_f64", "call": "host", "dtype": "f64", "n": 1 << 21, "recipe": "mixed64", "vectors": True},
        # Continuous-batching server: a burst of requests of uneven sizes, FP64 and compensated FP32.
        {"name": "serve", "call": "serve", "requests": 24, "largest": 1 << 18},
    ]


def _size(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["solve_f64", "values_f64", "solve_f32", "values_f32", "comp", "comp_ws", "comp_static", "train",
                       "bwd", "host", "serve"])
    # Slices of a larger batch start at any record: a call's input is then not always 16-byte aligned.
    skip = rng.choice([0, 0, 0, 1, 2, 3])
    if kind == "solve_f64":
        return {"call": "solve", "dtype": "f64", "n": _size(rng, 1, 1 << 23),
                "recipe": rng.choice(["mixed64", "spectral", "tensors"]), "vectors": True, "skip": skip}
    if kind == "values_f64":
        return {"call": "solve", "dtype": "f64", "n": _size(rng, 1, 1 << 23),
                "recipe": rng.choice(["mixed64_values", "spectral", "tensors"]), "vectors": False, "skip": skip}
    if kind in ("solve_f32", "values_f32"):
        return {"call": "solve", "dtype": "f32", "n": _size(rng, 1, 1 << 24),
                "recipe": rng.choice(["mixed32", "spectral", "tensors"]), "vectors": kind == "solve_f32", "skip": skip}
    if kind in ("comp", "comp_ws"):
        return {"call": kind, "dtype": "f32", "n": _size(rng, 1, 1 << 23),
                "recipe": rng.choice(["plane32", "mixed32", "tensors"]), "vectors": rng.random() < 0.8, "skip": skip}
    if kind == "comp_static":
        return {"call": kind, "dtype": "f32", "n": _size(rng, 1, syev3.STATIC_MAX_N), "recipe": "plane32",
                "vectors": True, "skip": skip}
    if kind == "train":
        return {"call": "train", "dtype": "f64", "n": _size(rng, 1, 1 << 21), "recipe": "spectral"}
    if kind == "bwd":
        return {"call": "bwd", "dtype": rng.choice(["f64", "f32"]), "n": _size(rng, 1, 1 << 22), "recipe": "spectral"}
    if kind == "host":
        dt = rng.choice(["f64", "f32"])
        return {"call": "host", "dtype": dt, "n": _size(rng, 1, 1 << 21),
                "recipe": "mixed64" if dt == "f64" else "mixed32", "vectors": rng.random() < 0.8}
    return {"call": "serve", "requests": _size(rng, 1, 32), "largest": _size(rng, 16, 1 << 18)}


def _torch_dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _repair(make, good, rounds=5):
    """make() with the rows that are not good() taken from further draws."""
    x = make()
    for _ in range(rounds):
        x = torch.where(good(x)[:, None], x, make())
    return x


def _rotation(q):
    """(m,4) quaternions -> (m,3,3) rotations, columns are the axes."""
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _no_tie(q):
    top = _rotation(q).abs().sort(dim=1, descending=True).values
    return ((top[:, 0] - top[:, 1]) > 1e-3).all(dim=1)


def _chunk(recipe, m, g):
    """m matrices: packed A (float64), their axes Q (columns) and values z
    before rounding, in the documented output order."""
    shares, ks, log_scale, kind, min_gap = RECIPES[recipe]
    dev = "cuda"
    opt = dict(generator=g, device=dev, dtype=torch.float64)

    def rand():
        return torch.rand(m, **opt)

    u = rand()
    edges = [sum(shares[:i + 1]) for i in range(5)]
    clustered = (u >= edges[0]) & (u < edges[1])
    near = (u >= edges[1]) & (u < edges[2])
    diagonal = (u >= edges[2]) & (u < edges[3])
    plane = u >= edges[3]

    def spectrum():
        z = torch.randn(m, 3, **opt)
        return 27.0 * torch.exp(0.3 * z) if kind == "positive" else z

    def apart(z):
        s = z.sort(dim=1).values
        return (s[:, 1:] - s[:, :-1]).amin(dim=1) >= min_gap * z.norm(dim=1)

    z = _repair(spectrum, apart)
    z = torch.where(apart(z)[:, None], z, torch.tensor([-1.0, 0.25, 1.0], device=dev, dtype=torch.float64))
    axes = _repair(lambda: torch.randn(m, 4, **opt), _no_tie)
    if shares[4] > 0:

        def in_plane():
            a, b = math.pi * rand(), math.pi * rand()
            ca, sa, cb, sb = a.cos(), a.sin(), b.cos(), b.sin()
            return torch.stack([ca * cb, ca * sb, sa * sb, sa * cb], 1)

        axes = torch.where(plane[:, None], _repair(in_plane, _no_tie), axes)
    Q = _rotation(axes)
    if shares[1] > 0:
        k = ks[0] + (ks[1] - ks[0]) * rand()
        zc = torch.stack([torch.ones_like(k), 1.0 + 10.0 ** (-k), -torch.ones_like(k)], 1)
        z = torch.where(clustered[:, None], zc, z)
    if shares[2] + shares[3] > 0:
        Q = torch.where((near | diagonal)[:, None, None], torch.eye(3, device=dev, dtype=torch.float64), Q)
        v, w, pat = torch.randn(m, **opt), torch.randn(m, **opt), (4 * rand()).floor()
        zr = torch.stack([torch.where(pat == 2, w, v), torch.where(pat == 1, w, v), torch.where(pat == 0, w, v)], 1)
        z = torch.where(diagonal[:, None], zr, z)
    z = z * 10.0 ** ((2.0 * rand() - 1.0) * log_scale)[:, None]
    A3 = (Q * z[:, None, :]) @ Q.transpose(1, 2)
    A = torch.stack([A3[:, 0, 0], A3[:, 1, 1], A3[:, 2, 2], A3[:, 0, 1], A3[:, 0, 2], A3[:, 1, 2]], 1)
    if shares[2] > 0:
        off = 1e-12 * torch.randn(m, 3, **opt) * z.norm(dim=1, keepdim=True)
        A[:, 3:] += torch.where(near[:, None], off, torch.zeros_like(off))
    # Ascending; equal values in the order of the first two by size, then the third.
    swap = z[:, 0] < z[:, 1]
    first = torch.tensor([0, 1, 2], device=dev)
    order = torch.where(swap[:, None], first[[1, 0, 2]], first)
    order = order.gather(1, z.gather(1, order).argsort(dim=1, stable=True))
    z = z.gather(1, order)
    Q = Q.gather(2, order[:, None, :].expand(-1, 3, -1))
    return A, Q, z


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)


def _chunks(recipe, n, g):
    for b in range(0, n, CHUNK):
        yield _chunk(recipe, min(CHUNK, n - b), g)


def _matrices(recipe, n, dtype, g, skip=0):
    """n packed matrices on the GPU, the slice after the first `skip` records."""
    big = torch.empty(n + skip, 6, dtype=dtype, device="cuda")
    big[:skip] = 0
    b = skip
    for A, _, _ in _chunks(recipe, n, g):
        big[b:b + A.shape[0]] = A
        b += A.shape[0]
    return big[skip:]


def _signed(Q):
    big = Q.gather(1, Q.abs().argmax(dim=1, keepdim=True))
    return Q * torch.where(big < 0, -1.0, 1.0)


def _eigenpairs(recipe, n, dtype, g):
    """Eigenvalues and eigenvectors in the solver's conventions, rounded to
    dtype; 5 % of the matrices with two values within 1e-9 of each other."""
    lam = torch.empty(n, 3, dtype=dtype, device="cuda")
    U = torch.empty(n, 3, 3, dtype=dtype, device="cuda")
    b = 0
    for _, Q, z in _chunks(recipe, n, g):
        m = z.shape[0]
        close = torch.rand(m, generator=g, device="cuda", dtype=torch.float64) < 0.05
        z[:, 1] = torch.where(close, z[:, 0] + 1e-9 * z.norm(dim=1), z[:, 1])
        lam[b:b + m] = z
        U[b:b + m] = _signed(Q)
        b += m
    return lam, U


def _requests(case):
    """The sizes of a burst, log-uniform up to the largest, and which are FP32."""
    r = case["requests"]
    return [(max(1, int(case["largest"] ** (((i * 7) % r + 1) / r))), i % 10 in (2, 5, 8)) for i in range(r)]


def prepare(case, seed):
    g = _generator(seed)
    call = case["call"]
    state = {"case": case}
    if call == "serve":
        state["server"] = syev3.Server(memory_budget_bytes=1 << 30)
        state["inputs"] = [(_matrices("plane32" if f32 else "mixed64", n, torch.float32 if f32 else torch.float64, g), f32)
                           for n, f32 in _requests(case)]
        return state
    n, dtype = case["n"], _torch_dtype(case)
    if call == "bwd":
        state["lam"], state["U"] = _eigenpairs(case["recipe"], n, dtype, g)
    elif call == "host":
        state["A"] = _matrices(case["recipe"], n, dtype, g).cpu().pin_memory()
        state["lam"] = torch.empty(n, 3, dtype=dtype, pin_memory=True)
        state["U"] = torch.empty(n, 3, 3, dtype=dtype, pin_memory=True) if case["vectors"] else None
    else:
        state["A"] = _matrices(case["recipe"], n, dtype, g, case.get("skip", 0))
    if call in ("train", "bwd"):
        state["gl"] = torch.randn(n, 3, generator=g, device="cuda", dtype=dtype)
        state["gU"] = torch.randn(n, 3, 3, generator=g, device="cuda", dtype=dtype)
    if call == "train":
        state["A"].requires_grad_(True)
    if call == "comp_ws":
        state["work"] = torch.empty(syev3.workspace_bytes(n, dtype, compensated=True), dtype=torch.uint8, device="cuda")
    return state


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "solve":
        return syev3.syev3_batched(state["A"], vectors=case["vectors"])
    if call == "comp":
        return syev3.syev3_batched(state["A"], vectors=case["vectors"], compensated=True)
    if call == "comp_ws":
        return syev3.syev3_batched(state["A"], vectors=case["vectors"], compensated=True, workspace=state["work"])
    if call == "comp_static":
        return syev3.syev3_batched_static_ws(state["A"], vectors=case["vectors"])
    if call == "train":
        lam, U = syev3.eigh3(state["A"])
        grad, = torch.autograd.grad((lam, U), state["A"], (state["gl"], state["gU"]))
        return lam.detach(), U.detach(), grad
    if call == "bwd":
        return syev3.syev3_batched_bwd(state["lam"], state["U"], state["gl"], state["gU"])
    if call == "host":
        return syev3.syev3_batched_host(state["A"], state["lam"], state["U"])
    server = state["server"]
    tickets = [server.submit(A, compensated=f32) for A, f32 in state["inputs"]]
    out = []
    for t in tickets:
        server.wait(t)
        lam, U = server.results(t)
        out.append((lam.clone(), U.clone()))
    torch.cuda.current_stream().synchronize()  # the results are copied before their memory goes back
    for t in tickets:
        server.release(t)
    return out


def work(case):
    call = case["call"]
    if call == "serve":
        return {"bytes": sum(n * (72 if f32 else 144) for n, f32 in _requests(case)),
                "flops": sum(n for n, _ in _requests(case)) * FLOPS}
    n, es = case["n"], 8 if case["dtype"] == "f64" else 4
    if call == "train":  # A, g_lambda, g_U in; lambda, U, the gradient out
        return {"bytes": n * es * (6 + 12 + 12 + 6), "flops": n * (FLOPS + FLOPS_BWD)}
    if call == "bwd":
        return {"bytes": n * es * 30, "flops": n * FLOPS_BWD}
    return {"bytes": n * es * (18 if case["vectors"] else 9), "flops": n * FLOPS}


def _exact_pairs(recipe, n, dtype, g):
    """Eigenpairs of the rounded matrices in 64 bits: perturbation to second
    order (values) and first order (vectors) about the construction's axes."""
    lams, Us = [], []
    for A, Q, _ in _chunks(recipe, n, g):
        A = A.to(dtype).double()
        A3 = A[:, [0, 3, 4, 3, 1, 5, 4, 5, 2]].view(-1, 3, 3)
        M = Q.transpose(1, 2) @ A3 @ Q
        d = M.diagonal(dim1=1, dim2=2)
        gap = d[:, None, :] - d[:, :, None]  # gap[j, i] = d_i - d_j
        off = M - torch.diag_embed(d)
        C = torch.where(off == 0, torch.zeros_like(off), off / gap)
        lams.append(d + (off * C).sum(dim=1))
        V = Q + Q @ C
        Us.append(_signed(V / V.norm(dim=1, keepdim=True)))
    return torch.cat(lams), torch.cat(Us)


def _exact_gradient(lam, U, gl, gU, tau=1e-6):
    lam, U, gl, gU = (t.double() for t in (lam, U, gl, gU))
    gap = lam[:, None, :] - lam[:, :, None]  # lambda_j - lambda_i at [i, j]
    masked = gap.abs() < tau * lam.norm(dim=1)[:, None, None]
    F = torch.where(masked, torch.zeros_like(gap), 1.0 / gap)
    G = U @ (torch.diag_embed(gl) + F * (U.transpose(1, 2) @ gU)) @ U.transpose(1, 2)
    S = G + G.transpose(1, 2)
    return torch.stack([G[:, 0, 0], G[:, 1, 1], G[:, 2, 2], S[:, 0, 1], S[:, 0, 2], S[:, 1, 2]], 1)


def exact(case, seed):
    g = _generator(seed)
    call = case["call"]
    if call == "serve":
        return [_exact_pairs("plane32" if f32 else "mixed64", n, torch.float32 if f32 else torch.float64, g)
                for n, f32 in _requests(case)]
    n, dtype = case["n"], _torch_dtype(case)
    if call == "bwd":
        state = prepare(case, seed)
        return _exact_gradient(state["lam"], state["U"], state["gl"], state["gU"])
    lam, U = _exact_pairs(case["recipe"], n, dtype, g)
    if call == "train":
        gl = torch.randn(n, 3, generator=g, device="cuda", dtype=dtype)
        gU = torch.randn(n, 3, 3, generator=g, device="cuda", dtype=dtype)
        return lam, U, _exact_gradient(lam, U, gl, gU)
    return lam, U if case["vectors"] else None
