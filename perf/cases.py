"""The work that a user of this library has it do, as measurable cases.

A case names one kind of call through the public entry points with its
sizes; `prepare` makes what a program has in hand before the call (the
handle, its preconditioner, the device blocks), `run` is the call, `work`
the bytes and operations one pass cannot do without, and `exact` the 64-bit
result of plain torch arithmetic where one exists.

Every field (variance, correlation length) and every input block is drawn
from the seed, so another seed is another operator as well as other inputs.
"""
import math

import numpy as np
import torch

import paper_2310_14649_gb300 as sg


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one small system (32^2 mesh, two random variables) solved to 1e-8:
        # a parameter study on a coarse mesh, where every launch counts
        dict(name="solve_32_p6", kind="solve", N=32, L=2, p=2, q=4, boxes=2, overlap=1, mode=1, tuned=True),
        # the ordinary solve: 256^2, four variables, 2.3M unknowns, mixed
        # precision, applies tuned once as a program that solves often does
        dict(name="solve_256_p35", kind="solve", N=256, L=4, p=3, q=6, boxes=8, overlap=2, mode=1, tuned=True),
        # the largest solve: 384^2, fourth-order chaos, 10.3M unknowns, the
        # defaults (no tuning)
        dict(name="solve_384_p70", kind="solve", N=384, L=4, p=4, q=8, boxes=16, overlap=2, mode=1, tuned=False),
        # the same system as the ordinary solve wholly in FP64
        dict(name="solve64_256_p35", kind="solve", N=256, L=4, p=3, q=6, boxes=8, overlap=2, mode=0, tuned=False),
        # four uneven systems in one graph launch (a family of fields)
        dict(name="batch_uneven", kind="batch", sizes="96:2:3:4,96:2:4:4,128:2:2:5,192:3:2:8"),
        # the operator alone, for a program with a Krylov method of its own
        dict(name="apply_256_p35", kind="apply", N=256, L=4, p=3, q=6, fp64=False, tuned=True),
        dict(name="apply_512_p84", kind="apply", N=512, L=6, p=3, q=6, fp64=False, tuned=False),
        # the restricted additive Schwarz smoother, the top kernel of a solve
        dict(name="smooth_256_p35", kind="smooth", N=256, L=4, p=3, q=6, boxes=8, overlap=2),
        # the coarse correction at the default inner tolerance (1e-5):
        # coarse GMRES, AMG cycles, coarse operator, transfers
        dict(name="coarse_256_p35", kind="coarse", N=256, L=4, p=3, q=6, boxes=8, overlap=2),
        # Newton's method for the nonlinear problem from a zero guess
        dict(name="newton_128_p35", kind="newton", N=128, L=4, p=3, q=6, boxes=5, overlap=2),
        # Monte Carlo verification samples, two full waves of the GPU
        dict(name="samples_100", kind="samples", N=100, L=3, S=304),
        # gradient of one training batch of the learned smoother
        dict(name="train_255_b32", kind="train", N=256, images=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _boxes(N):
    return int(min(max(round(N / 24), 2), 16))


# random variables and output order: 6 to 84 output terms (the input order
# is twice the output order, as in the shipped configurations)
_SMALL = [(2, 2), (2, 3), (3, 2), (2, 4), (4, 2), (3, 3), (5, 2)]
_MIDDLE = [(3, 4), (4, 3)]
_LARGE = [(5, 3), (4, 4), (6, 3)]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "apply", "apply", "apply", "smooth", "coarse", "newton",
                       "samples", "train"])
    if kind == "samples":
        return dict(kind=kind, N=_log_int(rng, 20, 102), L=rng.randint(1, 6), S=_log_int(rng, 8, 456))
    if kind == "train":
        return dict(kind=kind, N=2 * _log_int(rng, 16, 128), images=_log_int(rng, 4, 32))
    if kind == "batch":
        parts = []
        for _ in range(rng.randint(2, 5)):
            L, p = rng.choice(_SMALL)
            N = 2 * _log_int(rng, 24, 96)
            parts.append("%d:%d:%d:%d" % (N, L, p, _boxes(N)))
        return dict(kind=kind, sizes=",".join(parts))
    if kind == "apply":
        # meshes of either parity: the operator alone needs no coarse grid
        L, p = rng.choice(_SMALL + _MIDDLE + _LARGE)
        P = math.comb(L + p, p)
        N = _log_int(rng, 24, 400 if P <= 35 else 256)
        q = 2 * p
        fp64 = rng.random() < 0.3
        return dict(kind=kind, N=N, L=L, p=p, q=q, fp64=fp64, tuned=False)
    L, p = rng.choice(_SMALL + _MIDDLE)
    P = math.comb(L + p, p)
    if kind == "newton":
        N = 2 * _log_int(rng, 16, 64)
        return dict(kind=kind, N=N, L=L, p=p, q=2 * p, boxes=_boxes(N), overlap=rng.choice([1, 2]))
    N = 2 * _log_int(rng, 16, 160 if P <= 20 else 128)
    c = dict(kind=kind, N=N, L=L, p=p, q=2 * p, boxes=_boxes(N), overlap=rng.choice([1, 2]))
    if kind == "solve":
        c.update(mode=0 if rng.random() < 0.25 else 1, tuned=False)
    return c


# ---------------------------------------------------------------------------
# inputs from the seed
# ---------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _field(seed, salt=0):
    """Variance and correlation length of the lognormal field: those of the
    shipped configurations, each varied by a tenth."""
    r = np.random.default_rng([int(seed), 17 + salt])
    return dict(sigma2=float(0.3 * r.uniform(0.9, 1.1)), b=float(0.5 * r.uniform(0.9, 1.1)))


def _smooth_load(N, P, seed, salt=0):
    """Load block [P, n]: a smooth positive source in the mean, smaller
    smooth fluctuations in the first-order modes (P1 load, lumped)."""
    r = np.random.default_rng([int(seed), 29 + salt])
    m = N - 1
    t = torch.arange(1, N, device="cuda", dtype=torch.float64) / N
    F = torch.zeros((P, m * m), dtype=torch.float64, device="cuda")
    for a in range(min(P, 5)):
        f = torch.full((m, m), 1.0 if a == 0 else 0.0, dtype=torch.float64, device="cuda")
        for _ in range(4):
            kx, ky = r.integers(1, 5, 2)
            amp = r.uniform(-0.2, 0.2)
            f += amp * torch.cos(math.pi * ky * t)[:, None] * torch.cos(math.pi * kx * t)[None, :]
        F[a] = f.reshape(-1) / N ** 2
    return F


def _block(n, P, seed, salt, dtype):
    return torch.randn((P, n), generator=_gen(seed, salt), device="cuda", dtype=torch.float64).to(dtype)


def _setup(case, seed):
    f = _field(seed)
    return sg.sg_setup(case["N"], case["L"], case["p"], case["q"], sigma2=f["sigma2"], bx=f["b"], by=f["b"])


OMEGA = 0.3  # damping of the smoother case: found once, kept in the program


def _weights(seed):
    """He-normal weights and small biases of the five convolution layers."""
    r = np.random.default_rng([int(seed), 41])
    out = []
    for ci, co in zip(sg.CNN_CHANNELS[:-1], sg.CNN_CHANNELS[1:]):
        out.append((r.standard_normal((3, 3, ci, co)) * math.sqrt(2.0 / (9 * ci)), 0.05 * r.standard_normal(co)))
    return [(W.astype(np.float32), b.astype(np.float32)) for W, b in out]


def _train_pairs(N, images, seed):
    """Residual images and their targets: the target is smooth with some
    roughness, the residual the five-point Laplacian of it."""
    m = N - 1
    z = torch.randn((images, m, m), generator=_gen(seed, 5), device="cuda", dtype=torch.float32)
    for _ in range(3):
        z = torch.nn.functional.avg_pool2d(z[:, None], 3, 1, 1)[:, 0]
    zp = torch.nn.functional.pad(z, (1, 1, 1, 1))
    r = 4 * z - zp[:, :-2, 1:-1] - zp[:, 2:, 1:-1] - zp[:, 1:-1, :-2] - zp[:, 1:-1, 2:]
    return r.reshape(images, -1).contiguous(), z.reshape(images, -1).contiguous()


def _xi(case, seed):
    return torch.randn((case["S"], case["L"]), generator=_gen(seed, 3), device="cuda", dtype=torch.float64)


# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        probs, Xs, Fs = [], [], []
        for i, part in enumerate(case["sizes"].split(",")):
            N, L, p, boxes = (int(v) for v in part.split(":"))
            f = _field(seed, i + 1)
            pr = sg.sg_setup(N, L, p, 2 * p, sigma2=f["sigma2"], bx=f["b"], by=f["b"])
            sg.sg_precond_setup(pr, boxes, boxes, 2, inner_rtol=0.5, ras_kernel=0)
            probs.append(pr)
            Xs.append(torch.zeros((pr.P, pr.n), dtype=torch.float64, device="cuda"))
            Fs.append(_smooth_load(N, pr.P, seed, i + 1))
        return dict(case=case, batch=sg.sg_batch_create(probs, rtol=1e-8, mode=1), Xs=Xs, Fs=Fs)
    if kind == "samples":
        f = _field(seed)
        pr = sg.sg_setup(case["N"], case["L"], 2, 2, sigma2=f["sigma2"] / 30.0, bx=f["b"], by=f["b"])
        U = torch.zeros((case["S"], pr.n), dtype=torch.float32, device="cuda")
        return dict(case=case, prob=pr, xi=_xi(case, seed), U=U)
    if kind == "train":
        f = _field(seed)
        pr = sg.sg_setup(case["N"], 1, 1, 2, sigma2=f["sigma2"], bx=f["b"], by=f["b"])
        sg.sg_cnn_set_weights(pr, _weights(seed))
        R, Z = _train_pairs(case["N"], case["images"], seed)
        return dict(case=case, prob=pr, R=R, Z=Z)
    pr = _setup(case, seed)
    if case.get("tuned"):
        sg.sg_apply_autotune(pr)
    if kind == "apply":
        dt = torch.float64 if case["fp64"] else torch.float32
        X = _block(pr.n, pr.P, seed, 1, dt)
        return dict(case=case, prob=pr, X=X, Y=torch.zeros_like(X))
    s, ov = case["boxes"], case["overlap"]
    if kind == "smooth":
        sg.sg_precond_setup(pr, s, s, ov, omega=OMEGA, inner_rtol=0.5, ras_kernel=3)
        R = _block(pr.n, pr.P, seed, 1, torch.float32)
        return dict(case=case, prob=pr, R=R, Z=torch.zeros_like(R))
    if kind == "coarse":
        sg.sg_precond_setup(pr, s, s, ov, omega=OMEGA)
        R = _block(pr.n, pr.P, seed, 1, torch.float32)
        return dict(case=case, prob=pr, R=R, Z=torch.zeros_like(R))
    sg.sg_precond_setup(pr, s, s, ov, inner_rtol=0.5, ras_kernel=3)
    if case.get("tuned"):
        sg.sg_apply_autotune(pr, which=1)
    X = torch.zeros((pr.P, pr.n), dtype=torch.float64, device="cuda")
    if kind == "newton":
        return dict(case=case, prob=pr, X=X)
    return dict(case=case, prob=pr, X=X, F=_smooth_load(case["N"], pr.P, seed))


def run(s):
    kind = s["case"]["kind"]
    if kind == "solve":
        s["X"].zero_()
        sg.sg_solve(s["prob"], s["X"], F=s["F"], rtol=1e-8, mode=s["case"]["mode"])
        return {"X": s["X"]}
    if kind == "batch":
        for X in s["Xs"]:
            X.zero_()
        sg.sg_batch_solve(s["batch"], s["Xs"], s["Fs"])
        return {"X": list(s["Xs"])}
    if kind == "apply":
        sg.sg_apply(s["prob"], s["X"], s["Y"])
        return {"Y": s["Y"]}
    if kind == "smooth":
        sg.sg_precond_apply(s["prob"], sg.PC_SMOOTH, s["R"], s["Z"])
        return {"Z": s["Z"]}
    if kind == "coarse":
        sg.sg_precond_apply(s["prob"], sg.PC_COARSE, s["R"], s["Z"])
        return {"Z": s["Z"]}
    if kind == "newton":
        s["X"].zero_()
        sg.sg_newton(s["prob"], s["X"], tol_update=1e-8, mode=1)
        return {"X": s["X"]}
    if kind == "samples":
        sg.sg_sample_solve(s["prob"], s["xi"], s["U"], rtol=1e-6)
        return {"U": s["U"]}
    loss = sg.sg_cnn_train_step(s["prob"], s["R"], s["Z"], update=False)
    return {"loss": np.float32(loss), "grad": sg.sg_cnn_get_weights(s["prob"], gradient=True)}


# ---------------------------------------------------------------------------
# the bytes and operations one pass cannot do without
# ---------------------------------------------------------------------------
def _triples(L, p, q):
    """Number of nonzero <psi_k psi_a psi_b>."""
    return len(_triple_list(L, p, q)[0])


def _system_work(N, L, p, q, size, vecs):
    """One pass over the operator (a conductance per edge and input term)
    and `vecs` blocks of `size`-byte values; two operations per triple and
    edge, and the difference across and the scatter of each edge."""
    P, K, ne, n = math.comb(L + p, p), math.comb(L + q, q), 2 * N * (N - 1), (N - 1) ** 2
    return {"bytes": float(K * ne * size + vecs * n * P * size),
            "flops": float(2 * _triples(L, p, q) * ne + 3 * P * ne)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        out = {"bytes": 0.0, "flops": 0.0}
        for part in case["sizes"].split(","):
            N, L, p, _ = (int(v) for v in part.split(":"))
            w = _system_work(N, L, p, 2 * p, 8, 2)
            out = {k: out[k] + w[k] for k in out}
        return out
    if kind == "samples":
        n = (case["N"] - 1) ** 2
        # the samples and the solutions; one application of each sample's
        # operator at the least
        return {"bytes": float(8 * case["S"] * case["L"] + 4 * case["S"] * n + 16.0 * case["L"] * case["N"] ** 2),
                "flops": float(case["S"] * n * 10)}
    if kind == "train":
        pix = (case["N"] - 1) ** 2 * case["images"]
        c = sg.CNN_CHANNELS
        macs = sum(9 * a * b for a, b in zip(c[:-1], c[1:]))
        # forward, weight gradient, and input gradient of all but the first layer
        return {"bytes": float(8 * pix), "flops": float(2.0 * pix * (3 * macs - 9 * c[0] * c[1]))}
    N, L, p, q = case["N"], case["L"], case["p"], case["q"]
    if kind == "apply":
        return _system_work(N, L, p, q, 8 if case["fp64"] else 4, 2)
    P, n = math.comb(L + p, p), (N - 1) ** 2
    if kind == "smooth":
        # both blocks and the factors of the boxes' local matrices, banded
        # by lines (a line's width of values per node), once
        side = (N - 1) / case["boxes"] + 2 * case["overlap"]
        nodes = case["boxes"] ** 2 * side ** 2
        return {"bytes": float(8 * n * P + 4 * nodes * side), "flops": float(4 * nodes * side * P + 2 * n * P * P)}
    if kind == "coarse":
        w = _system_work(N // 2, L, p, q, 4, 0)
        return {"bytes": w["bytes"] + 8.0 * n * P, "flops": w["flops"] + 14.0 * n * P}
    # a solve: the operator, the right-hand side and the solution, once
    return _system_work(N, L, p, q, 8, 2)


# ---------------------------------------------------------------------------
# 64-bit results in plain torch
# ---------------------------------------------------------------------------
def _multi_indices(L, d):
    """Multi-indices of total degree <= d: by degree, then largest first."""
    out = []

    def rec(head, left, dims):
        if dims == 1:
            out.append(head + [left])
            return
        for v in range(left, -1, -1):
            rec(head + [v], left - v, dims - 1)

    for t in range(d + 1):
        rec([], t, L)
    return np.array(out)


def _he3(a, b, c):
    s, r = divmod(a + b + c, 2)
    if r or s < max(a, b, c):
        return 0
    f = math.factorial
    return f(a) * f(b) * f(c) // (f(s - a) * f(s - b) * f(s - c))


_TRIPLES = {}


def _triple_list(L, p, q):
    if (L, p, q) not in _TRIPLES:
        out, inp = _multi_indices(L, p), _multi_indices(L, q)
        t1 = np.array([[[_he3(k, a, b) for b in range(p + 1)] for a in range(p + 1)] for k in range(q + 1)], dtype=float)
        f = np.array([math.factorial(i) for i in range(max(p, q) + 1)], dtype=float)
        k, a, b, g = [], [], [], []
        fo = np.prod(f[out], axis=1)
        for i, al in enumerate(inp):
            v = np.ones((len(out), len(out)))
            for d in range(L):
                v = v * t1[al[d]][out[:, d][:, None], out[:, d][None, :]]
            ia, ib = np.nonzero(v)
            k.append(np.full(len(ia), i))
            a.append(ia)
            b.append(ib)
            g.append(v[ia, ib] / np.sqrt(np.prod(f[al]) * fo[ia] * fo[ib]))
        _TRIPLES[(L, p, q)] = tuple(np.concatenate(v) for v in (k, a, b, g))
    return _TRIPLES[(L, p, q)]


def _kl_modes(b, count):
    """1D eigenpairs of exp(-|s - t| / b) on [-1/2, 1/2]: (eigenvalue, frequency, odd)."""
    out = []
    for m in range(count):
        k = m // 2
        if m % 2 == 0:
            lo, hi, f = k * math.pi, k * math.pi + 0.5 * math.pi, lambda t: t * math.tan(t) - 0.5 / b
        else:
            lo, hi, f = k * math.pi + 0.5 * math.pi, (k + 1) * math.pi, lambda t: -t / math.tan(t) - 0.5 / b
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if mid <= lo or mid >= hi:
                break
            lo, hi = (mid, hi) if f(mid) < 0 else (lo, mid)
        w = 2.0 * lo
        out.append((2 * b / (1 + b * b * w * w), w, m % 2))
    return out


def _kl_phi(mode, s):
    _, w, odd = mode
    h = math.sin(w) / (2 * w)
    return torch.sin(w * s) / math.sqrt(0.5 - h) if odd else torch.cos(w * s) / math.sqrt(0.5 + h)


def _modes(N, L, sigma2, b):
    """g_i at the centroids of the lower and the upper triangles, [L, 2, N, N] (row j, column i)."""
    e = _kl_modes(b, L)
    pairs = sorted((-(sigma2 * (e[m][0] * e[n][0])), m, n) for m in range(L) for n in range(L))[:L]
    t = torch.arange(N, dtype=torch.float64, device="cuda")
    c1, c2 = (t + 1 / 3) / N - 0.5, (t + 2 / 3) / N - 0.5
    out = []
    for lam, m, n in pairs:
        lower = _kl_phi(e[n], c1)[:, None] * _kl_phi(e[m], c2)[None, :]
        upper = _kl_phi(e[n], c2)[:, None] * _kl_phi(e[m], c1)[None, :]
        out.append(math.sqrt(-lam) * torch.stack([lower, upper]))
    return torch.stack(out)


def _edges(c):
    """Edge conductances of a coefficient [..., 2, N, N]: horizontal
    [..., N-1, N] (rows j = 1..N-1), vertical [..., N, N-1]."""
    lo, up = c[..., 0, :, :], c[..., 1, :, :]
    return 0.5 * (lo[..., 1:, :] + up[..., :-1, :]), 0.5 * (up[..., :, 1:] + lo[..., :, :-1])


class _System:
    """The Galerkin system edge by edge: conductances of every input term
    made when they are needed, the triple products by input term."""

    def __init__(self, N, L, p, q, sigma2, b):
        self.N, self.P = N, math.comb(L + p, p)
        self.g = _modes(N, L, sigma2, b)
        self.c0 = torch.exp(0.5 * (self.g ** 2).sum(0))
        self.inp = _multi_indices(L, q)
        k, a, bb, g = _triple_list(L, p, q)
        self.by_k = {}
        for t in range(len(k)):
            self.by_k.setdefault(int(k[t]), []).append((int(a[t]), int(bb[t]), float(g[t])))

    def term(self, k):
        c = self.c0.clone()
        for i, d in enumerate(self.inp[k]):
            if d:
                c *= self.g[i] ** int(d) / math.sqrt(math.factorial(int(d)))
        return _edges(c)

    def apply(self, X):
        """sum_k A_k X G_k^T for X [P, n] in FP64."""
        m = self.N - 1
        x = torch.nn.functional.pad(X.double().reshape(self.P, m, m), (1, 1, 1, 1))
        dh = x[:, 1:-1, 1:] - x[:, 1:-1, :-1]
        dv = x[:, 1:, 1:-1] - x[:, :-1, 1:-1]
        fh, fv = torch.zeros_like(dh), torch.zeros_like(dv)
        for k, entries in self.by_k.items():
            wh, wv = self.term(k)
            for a, b, g in entries:
                fh[a].addcmul_(wh, dh[b], value=g)
                fv[a].addcmul_(wv, dv[b], value=g)
        y = fh[:, :, :-1] - fh[:, :, 1:] + fv[:, :-1, :] - fv[:, 1:, :]
        return y.reshape(self.P, m * m)

    def kronecker(self):
        """sum_k <A_k, A_0> / <A_0, A_0> G_k."""
        def diag(w):
            return w[0][:, :-1] + w[0][:, 1:] + w[1][:-1] + w[1][1:]

        w0 = self.term(0)
        d0 = diag(w0)

        def dot(w):
            return float((diag(w) * d0).sum() + 2 * (w[0][:, 1:-1] * w0[0][:, 1:-1]).sum()
                         + 2 * (w[1][1:-1] * w0[1][1:-1]).sum())

        G = torch.zeros((self.P, self.P), dtype=torch.float64, device="cuda")
        n0 = dot(w0)
        for k, entries in self.by_k.items():
            f = dot(self.term(k)) / n0
            for a, b, g in entries:
                G[a, b] += f * g
        return G

    def smooth(self, R, boxes, overlap, omega):
        """omega (G^-1 (x) I) sum_i R_i^T D_i (I (x) A_{0,i})^-1 R_i r."""
        m = self.N - 1
        wh, wv = self.term(0)
        diag = wh[:, :-1] + wh[:, 1:] + wv[:-1] + wv[1:]
        R = R.double()
        Z = torch.zeros_like(R)
        t = torch.arange(m, device="cuda")
        own = t * boxes // m
        owner = own[:, None] * boxes + own[None, :]
        for box in range(boxes * boxes):
            mem = owner == box
            for _ in range(overlap):
                q = torch.nn.functional.pad(mem, (1, 1, 1, 1))
                mem = q[1:-1, 1:-1] | q[:-2, 1:-1] | q[2:, 1:-1] | q[1:-1, :-2] | q[1:-1, 2:]
            idx = mem.reshape(-1).nonzero()[:, 0]
            place = torch.full((m * m,), -1, dtype=torch.long, device="cuda")
            place[idx] = torch.arange(len(idx), device="cuda")
            A = torch.diag(diag.reshape(-1)[idx])
            for step, w in ((1, wh[:, 1:-1]), (m, wv[1:-1])):
                full = torch.zeros((m, m), dtype=torch.float64, device="cuda")
                full[: w.shape[0], : w.shape[1]] = w
                has = (idx % m < m - 1) if step == 1 else (idx < m * (m - 1))
                i = idx[has]
                j = place[i + step]
                i = i[j >= 0]
                a, b = place[i], place[i + step]
                A[a, b] = A[b, a] = -full.reshape(-1)[i]
            z = torch.cholesky_solve(R[:, idx].T.contiguous(), torch.linalg.cholesky(A)).T
            mine = owner.reshape(-1)[idx] == box
            Z[:, idx[mine]] = z[:, mine]
        return omega * torch.linalg.solve(self.kronecker(), Z)


def _exact_samples(case, seed):
    """Conjugate gradients in FP64 on all samples to the rounding floor."""
    f = _field(seed)
    N, xi = case["N"], _xi(case, seed)
    g = _modes(N, case["L"], f["sigma2"] / 30.0, f["b"])
    m, wh, wv = N - 1, [], []
    for s in range(case["S"]):
        a, b = _edges(torch.exp(torch.tensordot(xi[s], g, 1)))
        wh.append(a)
        wv.append(b)
    wh, wv = torch.stack(wh), torch.stack(wv)
    dinv = 1.0 / (wh[:, :, :-1] + wh[:, :, 1:] + wv[:, :-1] + wv[:, 1:])

    def A(x):
        x = torch.nn.functional.pad(x, (1, 1, 1, 1))
        fh = wh * (x[:, 1:-1, 1:] - x[:, 1:-1, :-1])
        fv = wv * (x[:, 1:, 1:-1] - x[:, :-1, 1:-1])
        return fh[:, :, :-1] - fh[:, :, 1:] + fv[:, :-1] - fv[:, 1:]

    def dot(a, b):
        return (a * b).sum((1, 2), keepdim=True)

    r = torch.full((case["S"], m, m), 1.0 / N ** 2, dtype=torch.float64, device="cuda")
    x, z = torch.zeros_like(r), dinv * r
    p, rz, bb = z.clone(), dot(r, z), dot(r, r)
    for it in range(40 * N):
        q = A(p)
        alpha = rz / dot(p, q)
        x += alpha * p
        r -= alpha * q
        if it % 20 == 0 and bool((dot(r, r) <= 1e-24 * bb).all()):
            break
        z = dinv * r
        new = dot(r, z)
        p = z + new / rz * p
        rz = new
    return {"U": x.reshape(case["S"], m * m)}


def _exact_train(case, seed):
    """Loss (energy norm of A_0) and gradient of the network in FP64."""
    f = _field(seed)
    N, m = case["N"], case["N"] - 1
    R, Z = (t.double().reshape(-1, m, m) for t in _train_pairs(N, case["images"], seed))
    wh, wv = _edges(torch.exp(0.5 * (_modes(N, 1, f["sigma2"], f["b"]) ** 2).sum(0)))
    diag = wh[:, :-1] + wh[:, 1:] + wv[:-1] + wv[1:]
    params = []
    for W, b in _weights(seed):
        W = torch.tensor(W, dtype=torch.float64, device="cuda").requires_grad_()
        params += [W, torch.tensor(b, dtype=torch.float64, device="cuda").requires_grad_()]

    def energy(e):
        e = torch.nn.functional.pad(e, (1, 1, 1, 1))
        return ((wh * (e[:, 1:-1, 1:] - e[:, 1:-1, :-1]) ** 2).sum((1, 2))
                + (wv * (e[:, 1:, 1:-1] - e[:, :-1, 1:-1]) ** 2).sum((1, 2)))

    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    for i in range(0, len(R), 4):
        r, z = R[i:i + 4], Z[i:i + 4]
        rms = r.square().mean((1, 2), keepdim=True).sqrt()
        x = torch.stack([r / rms, torch.log(diag / 4).expand_as(r)], 1)
        for layer in range(5):
            # nine shifted products in place of a convolution call
            W, b = params[2 * layer], params[2 * layer + 1]
            xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
            x = b[None, :, None, None] + sum(
                torch.einsum("nchw,co->nohw", xp[:, :, dy:dy + m, dx:dx + m], W[dy, dx])
                for dy in range(3) for dx in range(3))
            if layer < 4:
                x = torch.relu(x)
        t = z / rms
        part = (energy(x[:, 0] - t) / energy(t)).sum()
        part.backward()
        loss += part.detach()
    grad = torch.cat([p.grad.reshape(-1) for p in params])
    return {"loss": float(loss), "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "samples":
        return _exact_samples(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind not in ("apply", "smooth", "solve"):
        return None
    f = _field(seed)
    N, L, p, q = case["N"], case["L"], case["p"], case["q"]
    n, P = (N - 1) ** 2, math.comb(L + p, p)
    S = _System(N, L, p, q, f["sigma2"], f["b"])
    if kind == "apply":
        return {"Y": S.apply(_block(n, P, seed, 1, torch.float64 if case["fp64"] else torch.float32))}
    if kind == "smooth":
        return {"Z": S.smooth(_block(n, P, seed, 1, torch.float32), case["boxes"], case["overlap"], OMEGA)}
    if n * P > 9000:
        return None
    # a small solve: the dense matrix column by column, solved directly
    A = torch.zeros((n * P, n * P), dtype=torch.float64, device="cuda")
    unit = torch.zeros((P, n), dtype=torch.float64, device="cuda")
    m = N - 1
    # nodes whose stencils do not meet share one application (spacing 3)
    t = torch.arange(m, device="cuda")
    for a in range(P):
        for sj in range(3):
            for si in range(3):
                pick = ((t % 3 == sj)[:, None] & (t % 3 == si)[None, :]).reshape(-1)
                unit.zero_()
                unit[a, pick] = 1.0
                y = S.apply(unit).reshape(P, m, m)
                for dj, di in ((0, 0), (0, 1), (0, -1), (1, 0), (-1, 0)):
                    src = pick.reshape(m, m).nonzero()
                    dst = src + torch.tensor([dj, di], device="cuda")
                    ok = ((dst >= 0) & (dst < m)).all(1)
                    src, dst = src[ok], dst[ok]
                    col = a * n + src[:, 0] * m + src[:, 1]
                    for bmode in range(P):
                        A[bmode * n + dst[:, 0] * m + dst[:, 1], col] = y[bmode, dst[:, 0], dst[:, 1]]
    F = _smooth_load(N, P, seed)
    return {"X": torch.linalg.solve(A, F.reshape(-1)).reshape(P, n)}
