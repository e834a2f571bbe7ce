"""What a program asks of this library, as cases to be measured.

Every case is one call through the public entry points, with the inputs of the
repository's own workloads (``synth/``, ``bench.py``): shifted Gaussian and
shifted uniform matrices, symmetric positive definite matrices with a
log-uniform spectrum, uneven batches of both, complex matrices.  The calls use
the library's defaults (tolerance 1e-12, automatic choice of the algorithm),
as a program that has read nothing but the signatures would.
"""
import math
import random

import torch

import paper_2607_12430_gb300 as mp


def listed():
    return [
        # the smallest sizes of the batch workload, solved one by one: a
        # covariance or coupling matrix of a small model, where launches and
        # host work are all there is
        {"name": "general-16", "call": "general", "n": 16, "dist": "gauss"},
        # an odd size below every tile of the large-matrix kernels
        {"name": "general-101", "call": "general", "n": 101, "dist": "gauss"},
        # the repository's benchmark matrix: 3I + G/sqrt(n)
        {"name": "general-512", "call": "general", "n": 512, "dist": "gauss"},
        # the nonsymmetric sets of the paper's Table 1 at their smaller size
        {"name": "uniform-2048", "call": "general", "n": 2048, "dist": "uniform"},
        # plain FP64 Schur method on a small SPD matrix: the accuracy run that
        # a program makes next to the mixed one
        {"name": "spd-fp64-64", "call": "fp64", "n": 64, "decades": 4},
        # an SPD matrix of ordinary, ragged size: whitening, a metric tensor
        {"name": "spd-777", "call": "spd", "n": 777, "decades": 4},
        # the large SPD workload of the benchmark, condition number 1e6
        {"name": "spd-4096", "call": "spd", "n": 4096, "decades": 6},
        # many matrices of uneven sizes in one call, half of them SPD
        {"name": "batch-2048", "call": "batch", "count": 2048, "lo": 16, "hi": 256},
        # a short batch of small matrices
        {"name": "batch-48", "call": "batch", "count": 48, "lo": 16, "hi": 96},
        # forward and backward of the differentiable square root
        {"name": "grad-256", "call": "grad", "n": 256},
        # complex input of odd size
        {"name": "complex-301", "call": "complex", "n": 301},
        # the principal cube root
        {"name": "cbrt-200", "call": "cbrt", "n": 200},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["general", "general", "general", "spd", "spd", "fp64", "batch", "batch", "grad", "complex", "cbrt"])
    if call == "general":
        return {"call": call, "n": _log_int(rng, 16, 2048), "dist": rng.choice(["gauss", "uniform"])}
    if call == "spd":
        return {"call": call, "n": _log_int(rng, 16, 4096), "decades": rng.choice([2, 4, 6])}
    if call == "fp64":
        return {"call": call, "n": _log_int(rng, 16, 512), "decades": rng.choice([2, 4])}
    if call == "batch":
        lo = _log_int(rng, 16, 64)
        return {"call": call, "count": _log_int(rng, 24, 2048), "lo": lo, "hi": _log_int(rng, lo + 8, 256)}
    if call == "grad":
        return {"call": call, "n": _log_int(rng, 16, 512)}
    return {"call": call, "n": _log_int(rng, 16, 512)}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _general(g, n, dist):
    """3I + G/sqrt(n), or U(0,1) entries and a shift that keeps every
    eigenvalue in the right half plane (the bulk of a U(0,1) matrix has
    spectral radius sqrt(n/12); a tenth more covers the edge eigenvalues)."""
    if dist == "gauss":
        A, shift = _normal(g, n, n) / math.sqrt(n), 3.0
    else:
        A = torch.rand(n, n, dtype=torch.float64, device="cuda", generator=g)
        shift = 1.1 * math.sqrt(n / 12.0) + 1.0
    A.diagonal().add_(shift)
    return A


def _spd(g, sizes, decades, pad):
    """Bitwise symmetric A = V diag(lam) V^T of every size, lam log-uniform
    over the decades around 1 with both ends taken: V is the Q of a Gaussian
    matrix, formed for all of them at once in blocks of pad x pad (a block's
    rest is the identity, which the factorisation keeps apart)."""
    ns = torch.tensor(sizes, device="cuda")[:, None]
    inside = torch.arange(pad, device="cuda")[None, :] < ns
    G = _normal(g, len(sizes), pad, pad) * (inside[:, :, None] & inside[:, None, :])
    G.diagonal(dim1=1, dim2=2).add_((~inside).double())
    V = torch.linalg.qr(G)[0]
    u = torch.rand(len(sizes), pad, dtype=torch.float64, device="cuda", generator=g)
    u[:, 0], u[:, 1] = 0.0, 1.0
    A = (V * (10.0 ** (decades * (u - 0.5)))[:, None, :]) @ V.mT
    A = 0.5 * (A + A.mT)
    return [A[i, :n, :n].contiguous() for i, n in enumerate(sizes)]


def _batch(g, count, lo, hi):
    """Sizes uniform in [lo, hi], the same ones for every seed; even members SPD
    over four decades, odd members 2I + G/sqrt(n)."""
    r = random.Random(f"{count} {lo} {hi}")
    sizes = [r.randint(lo, hi) for _ in range(count)]
    As = [None] * count
    for edge in range(32, 257, 32):
        members = [i for i in range(0, count, 2) if edge - 32 < sizes[i] <= edge]
        if members:
            for i, A in zip(members, _spd(g, [sizes[i] for i in members], 4, edge)):
                As[i] = A
    for i in range(1, count, 2):
        As[i] = _normal(g, sizes[i], sizes[i]) / math.sqrt(sizes[i])
        As[i].diagonal().add_(2.0)
    return As


def prepare(case, seed):
    g = _gen(seed)
    call = case["call"]
    s = {"call": call}
    if call == "general":
        s["A"] = _general(g, case["n"], case["dist"])
    elif call in ("spd", "fp64"):
        s["A"] = _spd(g, [case["n"]], case["decades"], case["n"])[0]
    elif call == "batch":
        s["As"] = _batch(g, case["count"], case["lo"], case["hi"])
        # the results side by side in one buffer, each on a 512-byte boundary
        step = [-(-A.numel() // 64) * 64 for A in s["As"]]
        s["flat"] = torch.zeros(sum(step), dtype=torch.float64, device="cuda")
        at = 0
        s["outs"] = []
        for A, k in zip(s["As"], step):
            s["outs"].append(s["flat"][at:at + A.numel()].view(A.shape))
            at += k
    elif call == "grad":
        s["A"] = _general(g, case["n"], "gauss").requires_grad_(True)
        s["G"] = _normal(g, case["n"], case["n"])
    elif call == "complex":
        n = case["n"]
        s["A"] = torch.complex(_normal(g, n, n), _normal(g, n, n)) / math.sqrt(2.0 * n)
        s["A"].diagonal().add_(3.0)
    elif call == "cbrt":
        s["A"] = _general(g, case["n"], "gauss")
    else:
        raise ValueError(call)
    return s


def run(state):
    call = state["call"]
    if call in ("general", "spd"):
        return mp.sqrtm_mixed(state["A"])[0]
    if call == "fp64":
        return mp.sqrtm_schur_fp64(state["A"])[0]
    if call == "batch":
        _, status = mp.sqrtm_mixed_batched(state["As"], outs=state["outs"])
        return {"roots": state["flat"], "failed": sum(1 for st in status if st)}
    if call == "grad":
        X = mp.sqrtm(state["A"])
        return {"root": X, "grad": torch.autograd.grad(X, state["A"], state["G"])[0]}
    if call == "complex":
        return mp.sqrtm_mixed_complex(state["A"])[0]
    return mp.cbrtm_mixed(state["A"])[0]


def work(case):
    """The matrix is read once and its root written once.  Operations: those
    of the Schur method in real arithmetic (Hessenberg form, Schur form with
    its vectors, triangular root, two products: 28 1/3 n^3), of the spectral
    method (tridiagonal form, its vectors, one symmetric product: 13/3 n^3),
    four times as many for complex matrices, and 10 n^3 for the gradient
    (four products and a triangular Sylvester solve)."""
    call = case["call"]
    if call == "batch":
        k, lo, hi = case["count"], case["lo"], case["hi"]
        n2 = k * sum(n ** 2 for n in range(lo, hi + 1)) / (hi - lo + 1)
        n3 = k * sum(n ** 3 for n in range(lo, hi + 1)) / (hi - lo + 1)
        return {"bytes": 16 * n2, "flops": (85 / 3 + 13 / 3) / 2 * n3}
    n = case["n"]
    if call in ("spd", "fp64"):
        return {"bytes": 16 * n * n, "flops": 13 / 3 * n ** 3}
    if call == "complex":
        return {"bytes": 32 * n * n, "flops": 4 * 85 / 3 * n ** 3}
    if call == "grad":
        return {"bytes": 32 * n * n, "flops": (85 / 3 + 10) * n ** 3}
    return {"bytes": 16 * n * n, "flops": 85 / 3 * n ** 3}


def _root_newton(A):
    """Principal square root of every matrix of a stack by the Denman-Beavers
    iteration with determinant scaling: the coupled iteration is stable and
    ends at rounding level."""
    n = A.shape[-1]
    Y, Z = A, torch.eye(n, dtype=A.dtype, device=A.device).expand_as(A)
    last = math.inf
    for k in range(40):
        if k < 8 and last > 1e-2:
            logdet = torch.linalg.slogdet(Y)[1] + torch.linalg.slogdet(Z)[1]
            mu = torch.exp(-logdet / (2.0 * n))[..., None, None]
        else:
            mu = 1.0
        Yi, Zi = torch.linalg.inv(Y), torch.linalg.inv(Z)
        Yn, Z = 0.5 * (mu * Y + Zi / mu), 0.5 * (mu * Z + Yi / mu)
        now = float(((Yn - Y).flatten(-2).norm(dim=-1) / Yn.flatten(-2).norm(dim=-1)).max())
        Y = Yn
        if now < 1e-13 or (now >= last and now < 1e-9):
            break
        last = now
    return Y


def _root_spectral(A):
    lam, V = torch.linalg.eigh(A)
    return (V * lam.sqrt()[..., None, :]) @ V.mT


def exact(case, seed):
    s = prepare(case, seed)
    call = case["call"]
    if call in ("spd", "fp64"):
        return _root_spectral(s["A"])
    if call in ("general", "complex"):
        return _root_newton(s["A"])
    if call == "cbrt":
        lam, V = torch.linalg.eig(s["A"].cpu())
        return ((V * lam.pow(1.0 / 3.0)[None, :]) @ torch.linalg.inv(V)).real.contiguous()
    if call == "grad":
        X = _root_newton(s["A"].detach()).cpu()
        G = s["G"].cpu()
        lam, V = torch.linalg.eig(X.mT)
        Vi = torch.linalg.inv(V)

        def solve(R):
            return (V @ ((Vi @ R.to(V.dtype) @ V) / (lam[:, None] + lam[None, :])) @ Vi).real

        Y = solve(G)
        Y = Y + solve(G - X.mT @ Y - Y @ X.mT)
        return {"root": X, "grad": Y}
    # batch: members of about the same size as one stack, each continued by
    # the identity, whose root is the identity
    for first in (0, 1):
        for edge in range(32, 257, 32):
            members = [i for i in range(first, len(s["As"]), 2) if edge - 32 < s["As"][i].shape[0] <= edge]
            if not members:
                continue
            B = torch.eye(edge, dtype=torch.float64, device="cuda").repeat(len(members), 1, 1)
            for k, i in enumerate(members):
                n = s["As"][i].shape[0]
                B[k, :n, :n] = s["As"][i]
            X = _root_spectral(B) if first == 0 else _root_newton(B)
            for k, i in enumerate(members):
                n = s["As"][i].shape[0]
                s["outs"][i].copy_(X[k, :n, :n])
    return {"roots": s["flat"], "failed": None}
