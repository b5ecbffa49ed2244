"""Performance cases of the framework: what its users run, through the public entry points.

A case is a dict with an operation (``op``), a point set (``data``, ``N``, ``beta``) and the operation's own sizes:

* ``apply``   one block product ``Y = M V`` of a context whose degrees are known (the call an outside solver makes once
  per iteration), in the fp32-grade or the reduced-precision mode;
* ``degree``  both degree passes at a bandwidth: q, d, s and the two off-diagonal sums;
* ``eigs``    a solve: degree passes and the leading k + 1 eigenpairs of M;
* ``flow``    the bandwidth flow over a new data set: context, probes, eigenpairs at the selected bandwidth;
* ``extend``  out-of-sample extension of known eigenvectors to new points.

Point sets (drawn on the GPU from the seed) have the shapes and bandwidths of the repository's own configurations: the
circle in R^2, the flat 2-torus in R^4, the noisy 6-torus in R^12, the anisotropic 6-torus zero-padded to R^32 and the
molecule-like latent torus in R^30.  The latent torus is one fixed system (its embedding does not depend on the seed) of
which every seed is another trajectory.
"""
import math

import numpy as np
import torch

import paper_2609_38198_b200 as fd

DIMS = {"circle": 2, "torus2": 4, "torus6": 12, "torus6pad": 32, "latent": 30}
RADII = (1.00, 1.08, 1.17, 1.27, 1.38, 1.50)
MEANS = ((-1.4, 2.6), (-1.4, -0.7), (1.1, -0.8), (-2.5, 2.9))
WEIGHTS = (0.4, 0.3, 0.2, 0.1)
KAPPA = 8.0


def listed():
    return [
        # the smallest call in use: a few thousand points in the plane, where launches and host latency count
        dict(name="circle_apply", op="apply", data="circle", N=2048, beta=200.0, b=8, prec="fp32"),
        # narrow kernel on a low-dimensional manifold (direct-difference kernels)
        dict(name="torus2_apply", op="apply", data="torus2", N=16384, beta=100.0, b=16, prec="fp32"),
        # a data set as it comes: ragged size, a block width that is no power of two
        dict(name="torus6_apply_odd", op="apply", data="torus6", N=50021, beta=2.0, b=20, prec="fp32"),
        # molecule-like trajectory: thirty coordinates, clustered two-dimensional latent space
        dict(name="latent_apply", op="apply", data="latent", N=262144, beta=2.0, b=32, prec="fp32"),
        # the headline product: a million points, 64 columns
        dict(name="torus6_apply_large", op="apply", data="torus6", N=1048576, beta=2.0, b=64, prec="fp32"),
        # the reduced-precision product of the precision cascade's first stage
        dict(name="torus6_apply_fast", op="apply", data="torus6", N=262144, beta=2.0, b=64, prec="fast"),
        # normalisation of a large data set: both degree passes
        dict(name="torus6_degree", op="degree", data="torus6", N=262144, beta=2.0),
        # a solve where the product is cheap and everything around it counts
        dict(name="torus2_eigs", op="eigs", data="torus2", N=16384, beta=30.0, k=32, b=16),
        # metastable modes of a trajectory: simple spectrum, ordinary size
        dict(name="latent_eigs", op="eigs", data="latent", N=65536, beta=2.0, k=32, b=32),
        # the large solve: 65 pairs of a clustered spectrum
        dict(name="torus6_eigs", op="eigs", data="torus6", N=131072, beta=2.0, k=64, b=32),
        # bandwidth selection on a small data set, from the raw points
        dict(name="torus6_flow", op="flow", data="torus6pad", N=8192, k=3, b=8),
        # extension of 33 eigenvectors to points that arrived later
        dict(name="latent_extend", op="extend", data="latent", N=65536, beta=2.0, M=40009, m=33),
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return n if rng.random() < 0.85 else max(lo, 1 << (n.bit_length() - 1))


def _beta(rng, data):
    lo, hi = {"circle": (50.0, 400.0), "torus2": (8.0, 300.0), "torus6": (0.25, 4.0), "latent": (0.5, 2.0)}[data]
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(("apply", "apply", "apply", "fast", "degree", "degree", "eigs", "eigs", "flow", "extend"))
    if op in ("apply", "fast"):
        data = rng.choice(("circle", "torus2", "torus6", "torus6", "latent")) if op == "apply" else rng.choice(("torus6", "latent"))
        lo, hi = {"circle": (1000, 20000), "torus2": (2000, 80000), "torus6": (3000, 500000), "latent": (4000, 300000)}[data]
        if op == "fast":
            lo = 16384
        return dict(op="apply", data=data, N=_log_int(rng, lo, hi), beta=_beta(rng, data), b=_log_int(rng, 1, 96),
                    prec="fp32" if op == "apply" else "fast")
    if op == "degree":
        data = rng.choice(("circle", "torus2", "torus6", "torus6", "latent"))
        lo, hi = {"circle": (1000, 20000), "torus2": (2000, 80000), "torus6": (3000, 500000), "latent": (4000, 300000)}[data]
        return dict(op="degree", data=data, N=_log_int(rng, lo, hi), beta=_beta(rng, data))
    if op == "eigs":
        data = rng.choice(("circle", "torus2", "torus6", "latent"))
        if data == "circle":
            return dict(op="eigs", data=data, N=_log_int(rng, 1500, 6000), beta=rng.uniform(100.0, 250.0), k=rng.choice((4, 8, 12)), b=8)
        if data == "torus2":
            return dict(op="eigs", data=data, N=_log_int(rng, 8000, 32000), beta=rng.uniform(8.0, 40.0), k=rng.randint(12, 36), b=16)
        if data == "torus6":
            return dict(op="eigs", data=data, N=_log_int(rng, 16384, 100000), beta=rng.uniform(0.5, 2.0), k=rng.randint(12, 64),
                        b=rng.choice((16, 32)))
        return dict(op="eigs", data=data, N=_log_int(rng, 8000, 100000), beta=rng.uniform(1.0, 2.0), k=rng.randint(8, 32),
                    b=rng.choice((16, 32)))
    if op == "flow":
        return dict(op="flow", data="torus6pad", N=_log_int(rng, 4100, 50000), k=rng.choice((3, 4, 6)), b=8)
    N = _log_int(rng, 8000, 120000)
    return dict(op="extend", data="latent", N=N, beta=_beta(rng, "latent"), M=_log_int(rng, 2000, 100000), m=rng.randint(4, 48))


def _points(data, N, seed, device):
    """N x D float32 points on the GPU, drawn in float64 and rounded once."""
    g = torch.Generator(device=device)
    g.manual_seed(1000003 * (seed + 1) + 17)

    def rand(*shape):
        return torch.rand(shape, generator=g, device=device, dtype=torch.float64)

    def randn(*shape):
        return torch.randn(shape, generator=g, device=device, dtype=torch.float64)

    if data == "circle":                                  # equispaced, from a random starting angle
        t = (torch.arange(N, device=device, dtype=torch.float64) / N + rand(1)) * (2.0 * math.pi)
        x = torch.stack([t.cos(), t.sin()], 1)
    elif data == "torus2":
        t = rand(N, 2) * (2.0 * math.pi)
        x = torch.stack([t.cos(), t.sin()], 2).reshape(N, 4)
    elif data in ("torus6", "torus6pad"):
        t = rand(N, 6) * (2.0 * math.pi)
        x = torch.stack([t.cos(), t.sin()], 2)
        if data == "torus6":
            x = x.reshape(N, 12) + 0.01 * randn(N, 12)
        else:
            x = (x * torch.tensor(RADII, device=device, dtype=torch.float64)[None, :, None]).reshape(N, 12)
            x = torch.cat([x, torch.zeros(N, 20, device=device, dtype=torch.float64)], 1)
    elif data == "latent":
        fixed = np.random.default_rng(42)                 # the system: the same for every trajectory
        W, c = fixed.standard_normal((30, 4)), fixed.standard_normal(30)
        rng = np.random.default_rng(seed + 1)
        comp = rng.choice(4, N, p=WEIGHTS)
        means = np.array(MEANS)
        a = torch.from_numpy(np.stack([rng.vonmises(means[comp, i], KAPPA) for i in (0, 1)], 1)).to(device)
        u = torch.stack([a.cos(), a.sin()], 2).reshape(N, 4)
        x = torch.tanh(u @ torch.from_numpy(W.T.copy()).to(device) + torch.from_numpy(c).to(device)) + 0.02 * randn(N, 30)
    else:
        raise ValueError(data)
    return x.to(torch.float32).contiguous()


def _block(N, b, seed, device):
    """N x b column-major block of i.i.d. N(0, 1) entries."""
    g = torch.Generator(device=device)
    g.manual_seed(7919 * (seed + 1) + 5)
    return torch.randn((b, N), generator=g, device=device, dtype=torch.float32).t()


def _basis_capacity(k, b):
    return 3 * (k + 1) + 2 * b


class State:
    def __init__(self, case, **kept):
        self.case = case
        self.__dict__.update(kept)


def prepare(case, seed):
    device = torch.device("cuda", torch.cuda.current_device())
    op, N = case["op"], case["N"]
    X = _points(case["data"], N, seed, device)
    if op == "apply":
        ctx = fd.Context(X, b_max=case["b"])
        prec = fd.FD_PREC_FAST if case["prec"] == "fast" else fd.FD_PREC_FP32
        ctx.degree(case["beta"], 1.0, prec=prec)
        return State(case, ctx=ctx, V=_block(N, case["b"], seed, device), prec=prec)
    if op == "degree":
        return State(case, ctx=fd.Context(X))
    if op == "eigs":
        k, b = case["k"], case["b"]
        # a direction of which every eigenvector has a component fixes the signs
        return State(case, ctx=fd.Context(X, b_max=b, m_max=_basis_capacity(k, b)), X=X, g=_block(N, 1, 12345, device))
    if op == "flow":
        return State(case, X=X)
    if op == "extend":
        every = _points(case["data"], N + case["M"], seed, device)
        X, Xnew = every[:N].contiguous(), every[N:].contiguous()
        ctx = fd.Context(X, b_max=64)
        ctx.degree(case["beta"], 1.0)
        # Smooth functions on the data set stand in for its eigenvectors: the extension treats any block alike.
        psi = torch.cos(X @ _block(30, case["m"], 99, device) * 0.3).t().contiguous().t()
        evals = [math.exp(-0.05 * j) for j in range(case["m"])]
        return State(case, ctx=ctx, Xnew=Xnew, psi=psi, evals=evals)
    raise ValueError(op)


def _smoothed(U, evals, X):
    """The points denoised by the leading part of the operator, U diag(evals) U^T X: what a spectral smoother keeps.
    Eigenvectors of a symmetric manifold come in clusters and are free to turn inside them; this is the same for all."""
    lam = torch.as_tensor(evals, dtype=torch.float32, device=X.device)
    return (U * lam) @ (U.t() @ X)


def run(state):
    c = state.case
    op = c["op"]
    if op == "apply":
        return state.ctx.apply(state.V, prec=state.prec)
    if op == "degree":
        return state.ctx.degree(c["beta"], 1.0)
    if op == "eigs":
        q, d, s, S_off, S_off2 = state.ctx.degree(c["beta"], 1.0)
        evals, U, info = state.ctx.eigs(c["k"], c["b"])
        if c["data"] == "latent":
            # a simple spectrum: the vectors themselves, with their signs fixed
            return evals, U * torch.sign(U.t() @ state.g).t()
        return evals, _smoothed(U, evals, state.X)
    if op == "flow":
        k, b = c["k"], c["b"]
        ctx = fd.Context(state.X, b_max=b, m_max=64)
        beta, outcome, evals, U, probes = ctx.beta_flow(k, b, 0.5)
        return beta, evals, np.array([p["V"] for p in probes]), _smoothed(U, evals, state.X)
    if op == "extend":
        return state.ctx.nystrom(state.Xnew, state.psi, state.evals)
    raise ValueError(op)


def work(case):
    """What one pass cannot do without: its inputs and outputs once, and per pair of points 2 D operations for the distance,
    one exponential and 2 per column of the product.  The degrees of a data set need each unordered pair once per pass."""
    op, N, D = case["op"], case["N"], DIMS[case["data"]]
    if op == "apply":
        b = case["b"]
        return {"bytes": 4.0 * N * (D + 2 * b + 1), "flops": float(N) * N * (2 * D + 1 + 2 * b)}
    degree = 2 * float(N) * N / 2 * (2 * D + 1 + 2)
    if op == "degree":
        return {"bytes": 4.0 * N * (D + 3), "flops": degree}
    if op == "eigs":
        # a Krylov space that holds k + 1 vectors: at least (k + 1) / b products
        n = math.ceil((case["k"] + 1) / case["b"])
        return {"bytes": 4.0 * N * (D + case["k"] + 1), "flops": degree + n * float(N) * N * (2 * D + 1 + 2 * case["b"])}
    if op == "flow":
        # three probes bracket a minimum and one is made at it; each needs its degrees and one product
        return {"bytes": 4.0 * N * (D + case["k"] + 1), "flops": 4 * (degree + float(N) * N * (2 * D + 1 + 2 * case["b"]))}
    M, m = case["M"], case["m"]
    return {"bytes": 4.0 * (N * (D + m + 1) + M * (D + m)), "flops": float(N) * M * (2 * D + 1 + 2 * (m + 1))}


def tolerance(case):
    """About four times what was measured: products, degrees and extensions against the same sums in float64 over direct
    differences, solves and flows against the same solve with another block width on the other kernels."""
    op, low = case["op"], DIMS[case["data"]] <= 4
    # in the plane and on the 2-torus the Gram form of the distance may serve only large sets at small bandwidths
    direct = low and (case["N"] < 16384 or case.get("beta", 0.0) > 25.0)
    if op == "apply":
        if case["prec"] == "fast":
            return {"rel": 1e-3}
        return {"rel": 1e-6 if direct else 1e-5 if low else 5e-6, "max": 4e-4}
    if op == "degree":
        return {"rel": 1e-6 if direct else 2e-5}
    if op == "extend":
        return {"rel": 2e-6}
    if op == "eigs":
        # single vectors of a simple spectrum move by residual / gap; what a cluster spans does not
        return {"rel": 1e-3} if case["data"] == "latent" else {"rel": 1e-5, "max": 4e-4}
    return {"rel": 2e-5}
