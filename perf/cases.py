"""The work a user has this framework do, as cases that can be timed and compared.

Every case is one call (or one training step) through the public Python entry points: a
vector OMT solve on an image grid, a matrix OMT solve on a tensor field, a complex Hermitian
solve, a solve on a volume, a batch of mixed problems, the differentiable transport cost with
its backward, and the unrolled gradient.  Sizes and options are those of the paper's tables,
of this repository's benchmark and tests, and the odd sizes that images and scans have.

Solves run a fixed number of iterations with their convergence checks every `check`
iterations (tolerances are never met), at a dual step tau of the size the tau tuner picks for
densities of unit mass, so that the fluxes are active and outputs can be compared.
"""
from __future__ import annotations

import itertools
import math
import random

import numpy as np
import torch

import paper_1712_10279_gb300 as V
from paper_1712_10279_gb300 import autograd

DEVICE = "cuda"
F64 = torch.float64

# --------------------------------------------------------------------------- the cases


def listed():
    return [
        # Table 1's smallest grid, colour blobs, one full solve of 2000 iterations: launches, checks and latency
        dict(name="vector_32_k3", kind="vector", n=32, k=3, graph="complete", alpha=1.0, iters=2000, check=100),
        # the colour-image solve of the benchmark (Table 1's largest grid)
        dict(name="vector_256_k3", kind="vector", n=256, k=3, graph="complete", alpha=0.1, iters=2000, check=100),
        # the paper's scalar comparison (Section 8.5): one channel, 1024 x 1024
        dict(name="scalar_1024", kind="vector", n=1024, k=1, graph="none", alpha=1.0, iters=500, check=100),
        # a photograph cropped to an odd size, regularised, joint norms
        dict(name="vector_601_k3_joint", kind="vector", n=601, k=3, graph="path", alpha=0.1, iters=300, check=50,
             u_norm="l2", w_norm="l2", eps=2.0e6),
        # the largest colour image: state beyond the L2 cache
        dict(name="vector_2048_k3", kind="vector", n=2048, k=3, graph="complete", alpha=0.1, iters=400, check=100),
        # the tensor-field solve of Table 3 (2-D DTI slice, 3 x 3 matrices, three L matrices)
        dict(name="matrix_128_3x3", kind="matrix", n=128, k=3, N=3, alpha=0.1, iters=1000, check=100),
        # multivariate spectral densities: 2 x 2 complex Hermitian fields
        dict(name="complex_96_2x2", kind="complex", n=96, k=2, N=3, alpha=0.1, iters=500, check=100),
        # a volume with three channels
        dict(name="volume_128_k3", kind="volume", n=128, k=3, graph="complete", alpha=0.3, iters=100, check=50),
        # a 3-D DTI volume of odd size, 3 x 3 tensors
        dict(name="tensor_volume_75_3x3", kind="tensor_volume", n=75, k=3, N=2, alpha=0.1, iters=60, check=30),
        # many small and middling problems of mixed size at once (pairwise distances of a data set)
        dict(name="batch_96_mixed", kind="batch", count=96, largest=256, mix=7, alpha=0.3, iters=300, check=100),
        # one training step on a batch of image pairs: transport cost and its envelope gradient
        dict(name="cost_step_8x256", kind="cost", batch=8, n=256, k=3, graph="complete", alpha=0.1, iters=500,
             check=100),
        # the gradient through an unrolled solve
        dict(name="unrolled_256_k3", kind="unrolled", n=256, k=3, graph="complete", alpha=0.1, T=200, ckpt=20),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; its cost stays below the largest listed one's."""
    kind = rng.choice(["vector", "vector", "vector", "matrix", "complex", "volume", "tensor_volume", "batch", "cost",
                       "unrolled"])
    alpha = round(math.exp(rng.uniform(math.log(0.05), math.log(1.0))), 3)
    check = rng.choice([20, 50, 100])
    if kind == "vector":
        k = rng.choice([1, 2, 3, 3, 3, 4, 5, 8])
        n = _log_int(rng, 16, 2048 if k <= 3 else 1024)
        case = dict(kind=kind, n=n, k=k, graph=_draw_graph(rng, k), alpha=alpha, check=check,
                    iters=check * max(1, min(20, int(3.0e9 / (n * n * (7 * k + k * (k - 1))) / check))),
                    u_norm=rng.choice(["l12", "l12", "l2", "l1"]), w_norm=rng.choice(["l1", "l1", "l2"]))
        if rng.random() < 0.2:
            case["eps"] = 5.0 * n * n
        return case
    if kind == "matrix":
        k, N = rng.choice([(2, 1), (2, 2), (2, 3), (3, 2), (3, 3)])
        n = _log_int(rng, 16, 512)
        return dict(kind=kind, n=n, k=k, N=max(N, 2), alpha=alpha, check=check,
                    iters=check * max(1, min(10, int(8.0e8 / (n * n * 30) / check))))
    if kind == "complex":
        return dict(kind=kind, n=_log_int(rng, 16, 160), k=2, N=rng.choice([2, 3]), alpha=alpha, check=check,
                    iters=check * rng.randint(2, 5))
    if kind == "volume":
        k = rng.choice([1, 3])
        n = _log_int(rng, 12, 144)
        return dict(kind=kind, n=n, k=k, graph=_draw_graph(rng, k), alpha=alpha, check=20,
                    iters=20 * max(1, min(10, int(3.0e9 / (n ** 3 * 9 * k) / 20))))
    if kind == "tensor_volume":
        k = rng.choice([2, 3])
        n = _log_int(rng, 12, 96)
        return dict(kind=kind, n=n, k=k, N=2, alpha=alpha, check=20,
                    iters=20 * max(1, min(5, int(2.0e9 / (n ** 3 * 60) / 20))))
    if kind == "batch":
        return dict(kind=kind, count=_log_int(rng, 4, 96), largest=rng.choice([64, 128, 256]),
                    mix=rng.randrange(1 << 16), alpha=alpha, check=check, iters=check * rng.randint(1, 3))
    if kind == "cost":
        k = rng.choice([1, 3])
        return dict(kind=kind, batch=rng.randint(1, 8), n=_log_int(rng, 24, 256), k=k, graph=_draw_graph(rng, k),
                    alpha=alpha, check=check, iters=check * rng.randint(1, 5))
    return dict(kind=kind, n=_log_int(rng, 24, 320), k=rng.choice([1, 3]), graph="complete", alpha=alpha,
                T=rng.randint(20, 150), ckpt=rng.choice([10, 20]))


def _draw_graph(rng, k):
    return "none" if k == 1 else rng.choice(["complete", "complete", "path"])


def _edges(k, graph):
    if k == 1 or graph == "none":
        return []
    if graph == "path":
        return [(a, a + 1) for a in range(k - 1)]
    return list(itertools.combinations(range(k), 2))


_U = {"l12": V.U_L12, "l2": V.U_L2, "l1": V.U_L1}
_W = {"l1": V.W_L1, "l2": V.W_L2}

# --------------------------------------------------------------------------- inputs


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _unit_mass(x):
    return x / x.sum()


def _blobs(r, k, shape, sigma, centre=(0.0, 1.0)):
    """Per channel three isotropic Gaussians and a small floor; centres in the given part of
    the grid; unit total mass."""
    axes = [torch.arange(n, device=DEVICE, dtype=F64) for n in shape]
    out = torch.full((k, *shape), 1e-3, device=DEVICE, dtype=F64)
    for c in range(k):
        for _ in range(3):
            s, a = r.uniform(*sigma), r.uniform(0.5, 1.0)
            term = torch.tensor(a, device=DEVICE, dtype=F64)
            for d, ax in enumerate(axes):
                g = torch.exp(-((ax - r.uniform(*centre) * shape[d]) ** 2) / (2.0 * s * s))
                term = term * g.reshape([-1 if e == d else 1 for e in range(len(shape))])
            out[c] += term
    return _unit_mass(out)


def _smooth(x, dims, sigma):
    """Gaussian filter with reflecting edges, one direction after the other."""
    radius = int(4.0 * sigma + 0.5)
    wt = [math.exp(-0.5 * (q / sigma) ** 2) for q in range(-radius, radius + 1)]
    total = sum(wt)
    for d in dims:
        n = x.shape[d]
        at = torch.arange(-radius, n + radius, device=x.device) % (2 * n)
        padded = x.index_select(d, torch.where(at < n, at, 2 * n - 1 - at))
        x = sum((v / total) * padded.narrow(d, q, n) for q, v in enumerate(wt))
    return x


def _image(r, g, n, k):
    """Smoothed noise and five rectangles of one colour each; unit total mass."""
    out = _smooth(torch.rand((k, n, n), generator=g, device=DEVICE, dtype=F64), (1, 2), 8.0)
    for _ in range(5):
        w, h = r.randint(min(8, n), min(64, n)), r.randint(min(8, n), min(64, n))
        x, y = r.randint(0, n - w), r.randint(0, n - h)
        for c in range(k):
            out[c, y:y + h, x:x + w] += r.uniform(0.5, 1.0)
    return _unit_mass(out)


def _unit_range(x):
    return (x - x.min()) / (x.max() - x.min())


def _tensors(g, k, shape, sigma, phase=False):
    """Q diag(lam) Q* with a smooth angle (and phase) field and smooth positive eigenvalues;
    unit total trace; [k*k, ...]."""
    dims = tuple(range(len(shape)))

    def noise():
        return _smooth(torch.rand(shape, generator=g, device=DEVICE, dtype=F64), dims, sigma)

    theta = 2.0 * math.pi * _unit_range(noise())
    lam = [0.05 + noise() for _ in range(k)]
    Q = torch.zeros((k, k, *shape), device=DEVICE, dtype=torch.complex128 if phase else F64)
    for a in range(k):
        Q[a, a] = 1.0
    Q[0, 0], Q[1, 1], Q[0, 1], Q[1, 0] = torch.cos(theta), torch.cos(theta), -torch.sin(theta), torch.sin(theta)
    if phase:
        turn = torch.exp(2j * math.pi * _unit_range(noise()))
        Q[0, 1], Q[1, 0] = Q[0, 1] * turn, Q[1, 0] * turn.conj()
    M = [sum(Q[a, e] * lam[e] * Q[b, e].conj() for e in range(k)) for a in range(k) for b in range(k)]
    return torch.stack(M) / sum(M[a * k + a].real.sum() for a in range(k))


def _L(seed, k, N, hermitian=False):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(N):
        G = rng.standard_normal((k, k))
        if hermitian:
            G = G + 1j * rng.standard_normal((k, k))
        S = 0.5 * (G + G.conj().T)
        out.append(S / np.linalg.norm(S))
    return np.stack(out)


def _tau(case):
    """The tuner's tau for densities of unit mass: it grows with the number of cells the
    mass is spread over (10 at 32 x 32, about 530 at 256 x 256 with three channels)."""
    dim = 3 if "volume" in case["kind"] else 2
    planes = case["k"] ** 2 if case["kind"] in ("matrix", "complex", "tensor_volume") else case["k"]
    return (0.003 if planes == case["k"] else 0.03) * planes * float(case["n"]) ** dim


def _mixed(case):
    """The problems of a batch (sides, channels and graphs), from the case alone."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        n = r.choice([s for s in (32, 64, 96, 128, 192, 256) if s <= case["largest"]])
        k = r.choice([1, 3, 5])
        edges = _edges(k, r.choice(["complete", "path"]))
        out.append(dict(n=n, k=k, edges=edges, alpha=case["alpha"], tau=0.003 * k * n * n))
    return out


def _inputs(case, seed):
    """The densities (float64) of a case; a list of pairs."""
    r, g, kind = random.Random(seed), _generator(seed), case["kind"]
    if kind == "batch":
        return [tuple(_blobs(r, p["k"], (p["n"],) * 2, (2.0, 5.0)) for _ in range(2)) for p in _mixed(case)]
    n, k = case["n"], case["k"]
    if kind in ("matrix", "complex"):
        return [tuple(_tensors(g, k, (n, n), min(10.0, n / 8.0), kind == "complex") for _ in range(2))]
    if kind == "tensor_volume":
        return [tuple(_tensors(g, k, (n, n, n), max(1.0, n / 12.0)) for _ in range(2))]
    if kind == "volume":
        return [tuple(_blobs(r, k, (n, n, n), (max(n / 12.0, 0.5), max(n / 5.0, 1.0))) for _ in range(2))]
    if n < 64:
        return [tuple(_blobs(r, k, (n, n), (2.0, 5.0)) for _ in range(2)) for _ in range(case.get("batch", 1))]
    return [tuple(_image(r, g, n, k) for _ in range(2)) for _ in range(case.get("batch", 1))]


def prepare(case, seed):
    kind = case["kind"]
    pairs = _inputs(case, seed)
    state = dict(case=case)
    if kind == "batch":
        state["batch"] = V.Batch(_mixed(case), [p[0].float() for p in pairs], [p[1].float() for p in pairs])
        return state
    if kind == "complex":
        state["rho"] = tuple(x.to(torch.complex64) for x in pairs[0])
    elif kind == "cost":
        state["rho"] = tuple(torch.stack([p[q] for p in pairs]).float() for q in range(2))
        state["alpha"] = torch.tensor(case["alpha"], device=DEVICE)
        state["weight"] = torch.rand(len(pairs), generator=_generator(seed + 1), device=DEVICE, dtype=F64) + 0.5
    else:
        state["rho"] = tuple(x.float() for x in pairs[0])
    if kind in ("matrix", "complex", "tensor_volume"):
        state["L"] = _L(seed, case["k"], case["N"], kind == "complex")
    return state


# --------------------------------------------------------------------------- one pass


def _numbers(result):
    return dict(primal=result["primal"], dual=result["dual"], iters=result["iters"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        bt = state["batch"]
        bt.solve(max_iters=case["iters"], check_every=case["check"])
        return dict(arena=bt.arena, primal=np.array([r["primal"] for r in bt.results], np.float32),
                    dual=np.array([r["dual"] for r in bt.results], np.float32))
    rho0, rho1 = state["rho"]
    if kind == "unrolled":
        J, d0, d1, da = autograd.unrolled_grad(rho0, rho1, _edges(case["k"], case["graph"]), case["alpha"],
                                               T=case["T"], ckpt=case["ckpt"], tau=_tau(case))
        return dict(J=J, d_rho0=d0, d_rho1=d1, d_alpha=da)
    many = dict(max_iters=case["iters"], check_every=case["check"], tau=_tau(case))
    if kind == "cost":
        r0, r1 = rho0.detach().requires_grad_(), rho1.detach().requires_grad_()
        alpha = state["alpha"].detach().requires_grad_()
        edges = _edges(case["k"], case["graph"])
        cost = autograd.transport_cost(r0, r1, edges, alpha, engine="batched", **many)
        loss = (state["weight"] * cost).sum()
        loss.backward()
        return dict(loss=loss.detach().float(), d_rho0=r0.grad, d_rho1=r1.grad, d_alpha=alpha.grad)
    if kind == "vector":
        sol = V.solve(rho0, rho1, _edges(case["k"], case["graph"]), case["alpha"], u_norm=_U[case.get("u_norm", "l12")],
                      w_norm=_W[case.get("w_norm", "l1")], eps=case.get("eps", 0.0), **many)
    elif kind == "volume":
        sol = V.solve3d(rho0, rho1, _edges(case["k"], case["graph"]), case["alpha"], **many)
    else:
        call = {"matrix": V.momt_solve, "complex": V.momt_solve_complex, "tensor_volume": V.momt_solve3d}[kind]
        sol = call(rho0, rho1, state["L"], case["alpha"], **many)
        return dict(U=sol.U, W=sol.W, Phi=sol.Phi, **_numbers(sol.result))
    return dict(u=sol.u, w=sol.w, phi=sol.phi, **_numbers(sol.result))


# --------------------------------------------------------------------------- work


def _point_flops(dim, channels, fluxes):
    """Arithmetic of one iteration at one point: per channel the gradient, the shrink, the
    extrapolation, the divergence and the ascent; per flux entry its gradient, shrink,
    extrapolation and divergence."""
    return channels * (13 * dim + 4) + fluxes * 13


def work(case):
    """Each input read once, each output written once; the arithmetic of every iteration."""
    kind = case["kind"]
    if kind == "batch":
        nbytes = flops = 0
        for p in _mixed(case):
            pts, k, l = p["n"] ** 2, p["k"], len(p["edges"])
            nbytes += 4 * pts * (5 * k + l)
            flops += case["iters"] * pts * _point_flops(2, k, l)
        return dict(bytes=nbytes, flops=flops)
    n, k, dim = case["n"], case["k"], 3 if "volume" in kind else 2
    pts = n ** dim * case.get("batch", 1)
    if kind in ("matrix", "tensor_volume"):
        planes = (2 + dim + 1 + case["N"]) * k * k
        return dict(bytes=4 * pts * planes,
                    flops=case["iters"] * pts * _point_flops(dim, k * (k + 1) // 2, case["N"] * k * (k - 1) // 2))
    if kind == "complex":
        return dict(bytes=8 * pts * (5 + case["N"]) * k * k,
                    flops=case["iters"] * pts * _point_flops(2, k * k, case["N"] * k * k))
    l = len(_edges(k, case["graph"]))
    flops = pts * _point_flops(dim, k, l)
    if kind == "unrolled":
        # forward once, reverse about twice the arithmetic of forward
        return dict(bytes=4 * pts * 4 * k, flops=3 * case["T"] * flops)
    if kind == "cost":
        return dict(bytes=4 * pts * 4 * k, flops=case["iters"] * flops)
    return dict(bytes=4 * pts * ((3 + dim) * k + l), flops=case["iters"] * flops)


# --------------------------------------------------------------------------- 64-bit results
# The iteration of Section 7 as plain torch operations in 64 bits.  Fields carry their
# components in front: phi [P, ...], u [dim, P, ...], w [M, ...], where P counts channels
# (matrix fields: the k*k entries) and M flux entries; G [M, P] is the matrix of the graph or
# quantum gradient and its divergence is -G^H.


def _forward(x, axis):
    """Difference to the next point along a grid axis; zero at the last one."""
    out = torch.zeros_like(x)
    m = x.shape[axis] - 1
    out.narrow(axis, 0, m).copy_(x.narrow(axis, 1, m) - x.narrow(axis, 0, m))
    return out


def _grad(phi, dim, ih):
    return torch.stack([ih * _forward(phi, phi.dim() - 1 - d) for d in range(dim)])


def _div(u, ih):
    """Backward differences (the ghost entries of u are zero)."""
    out = 0.0
    for d in range(u.shape[0]):
        axis = u.dim() - 2 - d
        m = u.shape[axis + 1] - 1
        back = u[d].clone()
        back.narrow(axis, 1, m).sub_(u[d].narrow(axis, 0, m))
        out = out + ih * back
    return out


def _apply(G, x):
    return (G @ x.reshape(x.shape[0], -1)).reshape(G.shape[0], *x.shape[1:])


def _norm(x, dims):
    return torch.sqrt((x * x.conj()).real.sum(dims, keepdim=True))


def _scale(x, dims, t):
    """The factor max(1 - t / |x|, 0), |x| the Euclidean norm over dims (one entry: ())."""
    s = _norm(x, dims) if dims else x.abs()
    pos = s > 0
    return torch.where(pos, torch.clamp(1.0 - t / torch.where(pos, s, torch.ones_like(s)), min=0.0),
                       torch.zeros_like(s))


_U_DIMS = {"l12": (0,), "l2": (0, 1), "l1": ()}
_W_DIMS = {"l2": (0,), "l1": ()}


class _Problem:
    def __init__(self, rho0, rho1, G, lmax, dim, tau, alpha, u_norm="l12", w_norm="l1", eps=0.0, matrix=False):
        n = rho0.shape[-1]
        self.b, self.G, self.dim, self.tau, self.alpha, self.eps = rho1 - rho0, G, dim, tau, alpha, eps
        self.ih = float(n - 1)
        share = 8.0 * dim if (G.shape[0] or matrix) else 4.0 * dim
        self.mu = 1.0 / (2.0 * share * tau * self.ih ** 2)
        self.nu = 1.0 / (4.0 * tau * lmax) if G.shape[0] else 1.0
        self.ud, self.wd = _U_DIMS[u_norm], _W_DIMS[w_norm]

    def start(self):
        z = torch.zeros_like(self.b)
        return z, torch.stack([z] * self.dim), z.new_zeros((self.G.shape[0], *z.shape[1:]))

    def step(self, phi, u, w, alpha=None):
        alpha = self.alpha if alpha is None else alpha
        su, sw = 1.0 / (1.0 + 2.0 * self.mu * self.eps), 1.0 / (1.0 + 2.0 * self.nu * self.eps)
        v = su * (u + self.mu * _grad(phi, self.dim, self.ih))
        u1 = v * _scale(v, self.ud, su * self.mu)
        r = _div(2.0 * u1 - u, self.ih) + self.b
        if self.G.shape[0]:
            x = sw * (w + self.nu * _apply(self.G, phi))
            w1 = x * _scale(x, self.wd, sw * alpha * self.nu)
            r = r - _apply(self.G.conj().T, 2.0 * w1 - w)
        else:
            w1 = w
        return phi + self.tau * r, u1, w1

    def primal(self, u, w, alpha=None):
        alpha = self.alpha if alpha is None else alpha
        P = (_norm(u, self.ud) if self.ud else u.abs()).sum()
        if w.shape[0]:
            P = P + alpha * (_norm(w, self.wd) if self.wd else w.abs()).sum()
        if self.eps:
            P = P + self.eps * ((u * u).sum() + (w * w).sum())
        return P

    def dual(self, phi):
        D = (phi * self.b.conj()).real.sum()
        if self.eps:
            for x, dims, radius in ((_grad(phi, self.dim, self.ih), self.ud, 1.0),
                                    (_apply(self.G, phi), self.wd, self.alpha)):
                if x.shape[0]:
                    s = _norm(x, dims) if dims else x.abs()
                    D = D - (torch.clamp(s - radius, min=0.0) ** 2).sum() / (4.0 * self.eps)
        return D

    def solve(self, iters):
        s = self.start()
        for _ in range(iters):
            s = self.step(*s)
        return s


def _graph_gradient(k, edges):
    G = np.zeros((len(edges), k))
    for e, (a, b) in enumerate(edges):
        G[e, min(a, b)], G[e, max(a, b)] = 1.0, -1.0
    return G, (float(np.linalg.eigvalsh(G.T @ G)[-1]) if edges else 0.0)


def _quantum_gradient(L):
    """X -> (L_s X - X L_s)_s on the k*k entries, row by row, and the largest eigenvalue of
    its Gram matrix over all k x k matrices."""
    k = L.shape[1]
    eye = np.eye(k)
    G = np.concatenate([np.kron(A, eye) - np.kron(eye, A.T) for A in L])
    return G, float(np.linalg.eigvalsh(G.conj().T @ G)[-1])


def _vector_problem(case, rho0, rho1, edges, tau):
    G, lmax = _graph_gradient(rho0.shape[0], edges)
    return _Problem(rho0, rho1, torch.tensor(G, device=DEVICE, dtype=F64), lmax, rho0.dim() - 1, tau, case["alpha"],
                    case.get("u_norm", "l12"), case.get("w_norm", "l1"), case.get("eps", 0.0))


def exact(case, seed):
    """What run() returns, in 64 bits, from the same (32-bit) densities."""
    kind = case["kind"]
    pairs = [tuple(x.to(torch.complex64 if kind == "complex" else torch.float32).to(
        torch.complex128 if kind == "complex" else F64) for x in p) for p in _inputs(case, seed)]
    if kind == "batch":
        probs = _mixed(case)
        chunks, P, D = [], [], []
        for p, (r0, r1) in zip(probs, pairs):
            prob = _vector_problem(case, r0, r1, p["edges"], p["tau"])
            phi, u, w = prob.solve(case["iters"])
            chunk = torch.cat([x.reshape(-1) for x in (r0, r1, u, w, phi)])
            pad = -chunk.numel() % 16
            chunks.append(torch.cat([chunk, chunk.new_zeros(pad)]))
            P.append(float(prob.primal(u, w)))
            D.append(float(prob.dual(phi)))
        return dict(arena=torch.cat(chunks), primal=np.array(P), dual=np.array(D))
    if kind == "unrolled":
        return _exact_unrolled(case, *pairs[0])
    if kind == "cost":
        weight = torch.rand(len(pairs), generator=_generator(seed + 1), device=DEVICE, dtype=F64) + 0.5
        loss, d_alpha, d1 = 0.0, 0.0, []
        for g, (r0, r1) in zip(weight.tolist(), pairs):
            prob = _vector_problem(case, r0, r1, _edges(case["k"], case["graph"]), _tau(case))
            phi, u, w = prob.solve(case["iters"])
            loss += g * float(prob.primal(u, w))
            d_alpha += g * float(w.abs().sum())
            d1.append(g * (phi - phi.mean()))
        d1 = torch.stack(d1)
        return dict(loss=torch.tensor(loss, dtype=F64), d_rho0=-d1, d_rho1=d1,
                    d_alpha=torch.tensor(d_alpha, dtype=F64))
    rho0, rho1 = pairs[0]
    if kind in ("vector", "volume"):
        prob = _vector_problem(case, rho0, rho1, _edges(case["k"], case["graph"]), _tau(case))
        phi, u, w = prob.solve(case["iters"])
        return dict(u=u, w=w, phi=phi, primal=float(prob.primal(u, w)), dual=float(prob.dual(phi)), iters=None)
    G, lmax = _quantum_gradient(_L(seed, case["k"], case["N"], kind == "complex"))
    kk = case["k"] ** 2
    prob = _Problem(rho0, rho1, torch.tensor(G, device=DEVICE, dtype=torch.complex128 if kind == "complex" else F64),
                    lmax, rho0.dim() - 1, _tau(case), case["alpha"], "l2", "l2" if kind == "complex" else "l1",
                    matrix=True)
    phi, u, w = prob.solve(case["iters"])
    return dict(U=u, W=w.reshape(case["N"], kk, *w.shape[1:]), Phi=phi, primal=float(prob.primal(u, w)),
                dual=float(prob.dual(phi)), iters=None)


def _exact_unrolled(case, rho0, rho1):
    if rho0.numel() * case["T"] > 1.2e8:
        return None
    rho1 = rho1.clone().requires_grad_()
    alpha = torch.tensor(case["alpha"], device=DEVICE, dtype=F64, requires_grad=True)
    prob = _vector_problem(case, rho0, rho1, _edges(case["k"], case["graph"]), _tau(case))
    s = tuple(x.detach() for x in prob.start())
    for _ in range(case["T"]):
        s = prob.step(*s, alpha=alpha)
    # the norm's derivative is taken as zero where the flux is zero
    u, w = s[1], s[2]
    n2 = (u * u).sum(0)
    J = torch.sqrt(torch.where(n2 > 0, n2, torch.ones_like(n2))).mul(n2 > 0).sum()
    J = J + alpha * w.abs().sum()
    d1, da = torch.autograd.grad(J, (rho1, alpha), allow_unused=True)
    return dict(J=J.detach(), d_rho0=-d1, d_rho1=d1, d_alpha=torch.zeros((), dtype=F64) if da is None else da)
