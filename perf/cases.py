"""Performance cases of the TTNS framework: what its users have it do, through its public calls.

A case is a dict of plain numbers and names.  Kinds:

  step     one tree advanced by ``steps`` sweeps, then rho_S and the occupations read
  batch    a batch of trees advanced by ``steps`` sweeps, populations left on the device
  observe  norm, energy, occupations, entropies and energy surfaces of an evolved tree
  train    one training step of the surrogate network (forward, backward, Adam)
  infer    one inference of the surrogate network

Spin-boson chains and the ER tree take the QR cutoff 1e-3 that the framework's own workloads
give them (at the default 1e-8 a long chain amplifies rounding within a few steps).

The mixed precision modes contract at the FP32 level, so a program keeps their results in
single precision (as the surrogate's data set does); FP64 results stay in double.

``exact`` restates the one-site TDVP sweep, its observables and the network in numpy / torch
float64, from the equations alone.
"""
import math

import numpy as np
import torch

from paper_1710_01362_gb300 import surrogate, ttns
from paper_1710_01362_gb300 import workloads as W

PRECISION = {"fp64": ttns.TTNS_FP64, "tf32x3": ttns.TTNS_TF32X3, "bf16x3": ttns.TTNS_BF16X3}
HBAR = 0.6582119569


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest run a user starts with: two states, an Ohmic chain of four sites, FP64
        dict(name="chain_4_fp64", kind="step", tree="chain", L=4, d=4, D=4, prec="fp64", cutoff=1e-3, steps=4, dt=0.5),
        # one ordinary spin-boson run at its truncated bonds, odd sizes
        dict(name="chain_25_tf32x3", kind="step", tree="chain", L=25, d=4, D=17, prec="tf32x3", cutoff=1e-3, steps=2,
             dt=0.5),
        # a small singlet-fission tree whose sites keep an optimised boson basis
        dict(name="star_3x6_obb_fp64", kind="step", tree="star", n_env=3, L=6, d=8, D=6, obb=4, prec="fp64",
             cutoff=0.0, steps=1, dt=0.5),
        # the star tree of the paper's shape: 5 states, 4 chains of 20 sites, in both precisions
        dict(name="star_4x20_tf32x3", kind="step", tree="star", n_env=4, L=20, d=10, D=20, obb=0, prec="tf32x3",
             cutoff=0.0, steps=1, dt=0.5),
        dict(name="star_4x20_fp64", kind="step", tree="star", n_env=4, L=20, d=10, D=20, obb=0, prec="fp64",
             cutoff=0.0, steps=1, dt=0.5),
        # the entanglement-renormalisation tree: the full headline run, and its short FP64 check
        dict(name="er_8x60_bf16x3", kind="step", tree="er", n_env=8, L=60, d=20, D=40, prec="bf16x3", cutoff=1e-3,
             steps=1, dt=0.25),
        dict(name="er_8x12_fp64", kind="step", tree="er", n_env=8, L=12, d=20, D=40, prec="fp64", cutoff=1e-3,
             steps=1, dt=0.25),
        # 256 spin-boson parameter sets advanced together (four CTAs per tree, as the benchmark does)
        dict(name="batch_256_tf32x3", kind="batch", tree="chain", n=256, ctas=4, prec="tf32x3", steps=1, dt=0.5),
        # training data of the surrogate: ER trees of eight short chains, one CTA per tree
        dict(name="surrogate_data_304_tf32x3", kind="batch", tree="surrogate", n=304, L=8, d=6, D=8, ctas=1,
             prec="tf32x3", steps=1, dt=1.0),
        # everything that is read from a tree during an analysis
        dict(name="observe_3x12_fp64", kind="observe", tree="star", n_env=3, L=12, d=8, D=12, obb=0, prec="fp64",
             cutoff=0.0, steps=6, dt=0.5),
        # one training step of the surrogate network at its batch size
        dict(name="train_256", kind="train", batch=256, points=200),
        # the held-out set answered by the network
        dict(name="infer_1000", kind="infer", batch=1000, points=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "star", "star", "er", "er", "batch", "surrogate", "observe", "train", "infer"])
    prec = rng.choice(["fp64", "tf32x3", "bf16x3"])
    if kind == "chain":
        return dict(kind="step", tree="chain", L=_log(rng, 3, 40), d=rng.randint(3, 8), D=rng.randint(3, 24), prec=prec,
                    cutoff=1e-3, steps=rng.randint(1, 4), dt=0.5)
    if kind == "star":
        n_env = rng.randint(2, 4)
        obb = rng.choice([0, 0, 0, rng.randint(3, 6)])
        return dict(kind="step", tree="star", n_env=n_env, L=_log(rng, 3, 20), d=rng.randint(4, 10),
                    D=rng.randint(5, 20), obb=obb, prec=prec, cutoff=0.0, steps=1, dt=0.5)
    if kind == "er":
        n_env = rng.choice([2, 4, 8])
        return dict(kind="step", tree="er", n_env=n_env, L=_log(rng, 3, 12 if prec == "fp64" else 24),
                    d=rng.randint(4, 20), D=rng.randint(6, 40), prec=prec, cutoff=1e-3, steps=1, dt=0.25)
    if kind == "batch":
        return dict(kind="batch", tree="chain", n=_log(rng, 16, 256), ctas=rng.choice([1, 2, 4, 8]), prec="tf32x3",
                    steps=1, dt=0.5)
    if kind == "surrogate":
        return dict(kind="batch", tree="surrogate", n=_log(rng, 32, 304), L=rng.randint(3, 8), d=rng.randint(4, 6),
                    D=rng.randint(5, 8), ctas=1, prec="tf32x3", steps=1, dt=1.0)
    if kind == "observe":
        return dict(kind="observe", tree="star", n_env=rng.randint(2, 3), L=_log(rng, 4, 14), d=rng.randint(4, 8),
                    D=rng.randint(6, 12), obb=0, prec="fp64", cutoff=0.0, steps=6, dt=0.5)
    if kind == "train":
        return dict(kind="train", batch=_log(rng, 32, 512), points=_log(rng, 20, 200))
    return dict(kind="infer", batch=_log(rng, 16, 2000), points=_log(rng, 20, 200))


# ------------------------------------------------------------------ inputs
def _problems(case, seed):
    """The Hamiltonians of a case: seeded draws of the framework's own workload generators."""
    t = case["tree"]
    if case["kind"] == "batch" and t == "chain":
        return [W.batched_spin_boson(1000 * (seed % 100000) + k) for k in range(case["n"])]
    if t == "surrogate":
        return [W.surrogate_problem(W.surrogate_params(1000 * (seed % 100000) + k), L=case["L"], d=case["d"],
                                    D=case["D"], dt=case["dt"]) for k in range(case["n"])]
    if t == "chain":
        r = np.random.default_rng(seed)
        p = W.spin_boson(eps=r.uniform(0.05, 0.15), V=r.uniform(0.02, 0.08), alpha=r.uniform(0.05, 0.3),
                         omega_c=r.uniform(0.1, 0.3), L=case["L"], d=case["d"], D=case["D"], dt=case["dt"])
    else:
        er = t == "er"
        modes = 2 * case["L"]
        p = W.singlet_fission(seed=seed, n_env=case["n_env"], L=case["L"], d=case["d"], D=case["D"], n_modes=modes,
                              dt=case["dt"], n_steps=case["steps"], er_tree=er, D_er=case["D"] if er else 0)
        for e in p.envs:
            e.obb = case.get("obb", 0)
    p.qr_cutoff = case["cutoff"] or None
    return [p]


def _training_set(case, seed):
    """Standardised parameter sets and smooth population trajectories."""
    r = np.random.default_rng(seed)
    n, pts = case["batch"], case["points"]
    X = np.stack([W.surrogate_params(int(s)) for s in r.integers(1 << 30, size=n)])
    X = (X - X.mean(axis=0)) / (X.std(axis=0) + 1e-12)
    t = np.arange(1, pts + 1) / pts
    w = r.uniform(2.0, 30.0, size=(n, 1, surrogate.N_STATES))
    Y = 1.0 + np.cos(w * t[None, :, None] + r.uniform(0, 6.3, size=(n, 1, surrogate.N_STATES)))
    Y = Y / Y.sum(axis=2, keepdims=True)
    return X, Y.reshape(n, -1)


def _widths(case):
    return [W.SURROGATE_N_PARAMS] + surrogate.WIDTHS_HIDDEN + [surrogate.N_STATES * case["points"]]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("train", "infer"):
        X, Y = _training_set(case, seed)
        return dict(case=case, net=surrogate.Net(_widths(case), seed),
                    x=torch.tensor(X, dtype=torch.float32, device="cuda"),
                    y=torch.tensor(Y, dtype=torch.float32, device="cuda"))
    ps = _problems(case, seed)
    kw = dict(precision=PRECISION[case["prec"]])
    if kind == "batch":
        tree = ttns.Tree(ps, cluster_ctas=case["ctas"], **kw)
        out = torch.zeros(sum(p.n_el for p in ps), dtype=torch.float64, device="cuda")
        return dict(case=case, tree=tree, out=out)
    tree = ttns.Tree(ps[0], **kw)
    if kind == "observe":
        tree.step(case["dt"], case["steps"])
        tree.sync()
    return dict(case=case, tree=tree)


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "train":
        net = state["net"]
        y, hs = net.forward(state["x"])
        grads = net.backward(hs, y, state["y"])
        net.adam(grads, 1e-3)
        return dict(y=y, dW=[g[0] for g in grads], db=[g[1] for g in grads], m=list(net.mW), v=list(net.vW),
                    W=list(net.W), b=list(net.b))
    if kind == "infer":
        y, _ = state["net"].forward(state["x"], kind=surrogate.KIND_INFER)
        return dict(y=y)
    tree = state["tree"]
    if kind == "observe":
        norm, energy = tree.observables()
        tes, pes, sigma = tree.energy_surfaces()
        return dict(rho=tree.rho(), norm=norm, energy=energy, occ=tree.occupations(), entropy=tree.bond_entropies(),
                    tes=tes, pes=pes, sigma=sigma)
    tree.step(case["dt"], case["steps"])
    if kind == "batch":
        tree.populations_device(state["out"].data_ptr())
        return dict(pop=state["out"].float())
    rho, occ = tree.rho(), tree.occupations()
    if case["prec"] != "fp64":
        rho, occ = rho.astype(np.complex64), occ.astype(np.float32)
    return dict(rho=rho, occ=occ)


# ------------------------------------------------------------------ the tree (shapes and operators)
class _Tree:
    """Nodes in creation order (root 0), legs [parent][children][physical], clamped bonds, and
    the Hamiltonian's terms: on-site operators and products of two single-node operators."""

    def __init__(self, p):
        self.parent, self.children, self.phys, req = [], [], [], []

        def add(par, ph, D):
            v = len(self.parent)
            self.parent.append(par)
            self.children.append([])
            self.phys.append(ph)
            req.append(D)
            if par >= 0:
                self.children[par].append(v)
            return v

        add(-1, p.n_el, 0)
        ends = [0] * len(p.envs)
        if p.er_tree:
            level = [add(0, 0, p.D_er)]
            while 2 * len(level) < len(p.envs):
                level = [add(v, 0, p.D_er) for v in level for _ in range(2)]
            ends = [v for v in level for _ in range(2)]
        self.sites = []
        for e, v in zip(p.envs, ends):
            chain = []
            for _ in range(e.L):
                v = add(v, 0 if e.obb else e.d, e.D)
                chain.append(add(v, e.d, e.obb) if e.obb else v)
            self.sites.append(chain)
        self.n = len(self.parent)
        self.bond = req
        while True:  # every bond at most the product of the other legs, at both of its ends
            old = list(self.bond)
            for u in range(1, self.n):
                v = self.parent[u]
                at_v = [self.bond[v]] * (v > 0) + [self.bond[c] for c in self.children[v] if c != u]
                lim = [math.prod([max(self.phys[u], 1)] + [self.bond[c] for c in self.children[u]]),
                       math.prod([max(self.phys[v], 1)] + at_v)]
                self.bond[u] = min([self.bond[u]] + lim)
            if old == self.bond:
                break
        self.sub = [{v} for v in range(self.n)]
        for v in range(self.n - 1, 0, -1):
            self.sub[self.parent[v]] |= self.sub[v]

    def dims(self, v):
        return [self.bond[v]] * (v > 0) + [self.bond[c] for c in self.children[v]] + [self.phys[v]] * (self.phys[v] > 0)

    def leg(self, v, u):
        if self.parent[v] == u:
            return 0
        return (v > 0) + self.children[v].index(u)

    def near(self, v):
        return [self.parent[v]] * (v > 0) + self.children[v]

    def toward(self, v, x):
        return next((c for c in self.children[v] if x in self.sub[c]), self.parent[v])

    def side(self, u, v, x):
        """Whether node x is on u's side of the edge (u, v)."""
        return x in self.sub[u] if self.parent[u] == v else x not in self.sub[v]


def _chain_of(e):
    if e.spectral[0] == "ohmic":
        _, alpha, wc = e.spectral
        k = np.arange(e.L)
        return 2 * wc * math.sqrt(alpha), wc * (2 * k + 2), wc * np.sqrt((k[:-1] + 1.0) * (k[:-1] + 2.0))
    w, lam = np.asarray(e.spectral[1], float), np.asarray(e.spectral[2], float)
    rc = np.linalg.norm(lam)
    Q, on, hop = [lam / rc], [], []
    for k in range(e.L):
        x = w * Q[k]
        on.append(Q[k] @ x)
        for _ in range(2):
            x = x - np.array(Q).T @ (np.array(Q) @ x)
        if k + 1 < e.L:
            hop.append(np.linalg.norm(x))
            Q.append(x / hop[-1])
    return rc, np.array(on), np.array(hop)


def _operators(p, t, kinetic=False):
    """(on-site operators, two-node terms) of the Hamiltonian, or of the chains' kinetic energy."""
    onsite, terms = [None] * t.n, []
    if not kinetic:
        onsite[0] = p.H_S - np.trace(p.H_S).real / p.n_el * np.eye(p.n_el)
    for e, nodes in zip(p.envs, t.sites):
        rc, on, hop = _chain_of(e)
        a = np.diag(np.sqrt(np.arange(1.0, e.d)), 1).astype(complex)
        up = a.T.copy()
        for k, v in enumerate(nodes):
            onsite[v] = -0.25 * on[k] * (up - a) @ (up - a) if kinetic else on[k] * (up @ a)
        if not kinetic:
            terms.append((0, rc / math.sqrt(2) * p.W_of(e), nodes[0], a + up))
        for k in range(e.L - 1):
            if kinetic:
                terms.append((nodes[k], -0.5 * hop[k] * (up - a), nodes[k + 1], up - a))
            else:
                terms += [(nodes[k], hop[k] * up, nodes[k + 1], a), (nodes[k], hop[k] * a, nodes[k + 1], up)]
    return onsite, terms


# ------------------------------------------------------------------ the sweep in FP64 numpy
def _on(M, A, l):
    """M applied on leg l of A."""
    s = A.shape
    X = A.reshape(math.prod(s[:l]), s[l], -1)
    return np.matmul(M, X).reshape(s[:l] + (M.shape[0],) + s[l + 1:])


def _over(Q, X, l):
    """sum over every leg but l of conj(Q) X."""
    q, x = np.moveaxis(Q, l, 0), np.moveaxis(X, l, 0)
    return q.reshape(q.shape[0], -1).conj() @ x.reshape(x.shape[0], -1).T


def _qr(M, cutoff):
    """Householder QR: a sub-column of norm <= cutoff |M| is dropped and takes the identity
    reflector; the diagonal of R is real and >= 0; R is scaled back to |M|."""
    m, n = M.shape
    X, fro, vs = M.astype(complex), np.linalg.norm(M), []
    R = np.zeros((n, n), complex)
    for j in range(n):
        x = X[j:, j].copy()
        s = np.linalg.norm(x)
        v = None
        if s > cutoff * fro:
            ph = x[0] / abs(x[0]) if abs(x[0]) > 1e-280 else 1.0
            R[j, j] = -ph * s
            x[0] += ph * s
            v = x / np.linalg.norm(x)
            X[j:, j + 1:] -= np.outer(2 * v, v.conj() @ X[j:, j + 1:])
        vs.append(v)
        R[j, j + 1:] = X[j, j + 1:]
    Q = np.eye(m, n, dtype=complex)
    for j in range(n - 1, -1, -1):
        if vs[j] is not None:
            Q[j:] -= np.outer(2 * vs[j], vs[j].conj() @ Q[j:])
    ph = np.array([R[j, j] / abs(R[j, j]) if R[j, j] != 0 else 1.0 for j in range(n)])
    Q, R = Q * ph, R * ph.conj()[:, None]
    k = np.linalg.norm(R)
    return Q, R * (fro / k) if k else R


def _expm(apply, x, s):
    """exp(-i s H) x on Krylov spaces of dimension <= 30, to 1e-14; the time is halved until it fits."""
    shape, y = x.shape, x.reshape(-1).astype(complex)
    while s:
        b0 = np.linalg.norm(y)
        K, al, be = [y / b0], [], []
        done = False
        while True:
            w = apply(K[-1].reshape(shape)).reshape(-1)
            al.append(np.vdot(K[-1], w).real)
            B = np.array(K)
            for _ in range(2):
                w = w - B.T @ (B.conj() @ w)
            b = np.linalg.norm(w)
            ev, S = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
            u = S @ (np.exp(-1j * s * ev) * S[0])
            done = b * abs(u[-1]) <= 1e-14 or len(al) == y.size
            if done or len(al) == 30:
                break
            be.append(b)
            K.append(w / b)
        h = s
        while not done and b * abs(u[-1]) > 1e-14:
            h /= 2
            u = S @ (np.exp(-1j * h * ev) * S[0])
        y = b0 * (u @ np.array(K))
        s = s - h
    return y.reshape(shape)


class _Sweep:
    def __init__(self, p):
        p.W_of = lambda e: np.asarray(e.W_bar, complex)
        self.p, self.t = p, _Tree(p)
        t = self.t
        self.ops = _operators(p, t)
        self.A = []
        for v in range(t.n):
            s = t.dims(v)
            if v:
                self.A.append(np.eye(s[0], math.prod(s[1:]), dtype=complex).reshape(s))
            else:
                A = np.zeros(s, complex)
                A[(0,) * (len(s) - 1) + (p.init_state,)] = 1.0
                self.A.append(A)
        self.env = {}
        for v in range(t.n - 1, 0, -1):
            self.update(v, t.parent[v])

    def end(self, v, x, op, k):
        """(leg, matrix) of term k's end at node x, seen from node v."""
        if x == v:
            return len(self.t.dims(v)) - 1, op
        w = self.t.toward(v, x)
        return self.t.leg(v, w), self.env[w, v][1 + k]

    def heff(self, v, x, without=None):
        t, (onsite, terms) = self.t, self.ops
        one = {}  # single-leg terms, added up per leg
        if onsite[v] is not None:
            one[len(t.dims(v)) - 1] = onsite[v]
        for w in t.near(v):
            if w != without:
                one[t.leg(v, w)] = one.get(t.leg(v, w), 0) + self.env[w, v][0]
        y = sum((_on(M, x, l) for l, M in one.items()), np.zeros_like(x))
        for k, (a, oa, b, ob) in enumerate(terms):
            if without is not None and not (t.side(v, without, a) and t.side(v, without, b)):
                continue
            if (v if a == v else t.toward(v, a)) != (v if b == v else t.toward(v, b)):
                (la, Ma), (lb, Mb) = self.end(v, a, oa, k), self.end(v, b, ob, k)
                y += _on(Mb, _on(Ma, x, la), lb)
        return y

    def update(self, u, v):
        t, Q, l = self.t, self.A[u], self.t.leg(u, v)
        E = {0: _over(Q, self.heff(u, Q, v), l)}
        for k, (a, oa, b, ob) in enumerate(self.ops[1]):
            ina, inb = t.side(u, v, a), t.side(u, v, b)
            if ina != inb:
                m, M = self.end(u, a if ina else b, oa if ina else ob, k)
                E[1 + k] = _over(Q, _on(M, Q, m), l)
        self.env[u, v] = E

    def hbond(self, u, w, X):
        E, F = self.env[u, w], self.env[w, u]
        return E[0] @ X + X @ F[0].T + sum(E[k] @ X @ F[k].T for k in E if k)

    def forward(self, v, tau):
        self.A[v] = _expm(lambda x: self.heff(v, x), self.A[v], tau / HBAR)

    def move(self, v, u, tau):
        """The centre from v to u; the bond evolves backward by tau when tau is not 0."""
        t, l = self.t, self.t.leg(v, u)
        X = np.moveaxis(self.A[v], l, -1)
        Q, R = _qr(X.reshape(-1, X.shape[-1]), self.p.qr_cutoff or 1e-8)
        self.A[v] = np.moveaxis(Q.reshape(X.shape), -1, l)
        self.update(v, u)
        if tau:
            R = _expm(lambda x: self.hbond(v, u, x), R, -tau / HBAR)
        self.A[u] = _on(R, self.A[u], t.leg(u, v))

    def down(self, v, tau):
        self.forward(v, tau)
        for c in self.t.children[v]:
            self.move(v, c, tau)
            self.down(c, tau)
            self.move(c, v, 0)

    def up(self, v, tau):
        for c in reversed(self.t.children[v]):
            self.move(v, c, 0)
            self.up(c, tau)
            self.move(c, v, tau)
        self.forward(v, tau)

    def step(self, dt, n):
        for _ in range(n):
            self.down(0, dt / 2)
            self.up(0, dt / 2)

    def rho(self):
        A = self.A[0]
        return _over(A.conj(), A.conj(), A.ndim - 1)

    def densities(self):
        """(density of every bond, occupation of every site), from the root down."""
        t, bond, occ = self.t, {}, {}
        for v in range(t.n):
            Q = self.A[v]
            X = _on(bond[v].T, Q, 0) if v else Q
            for c in t.children[v]:
                bond[c] = _over(Q, X, t.leg(v, c)).T
            if v and t.phys[v]:
                r = _over(Q, X, Q.ndim - 1)
                occ[v] = float(np.arange(len(r)) @ np.diag(r).real)
        return bond, np.array([occ[v] for chain in t.sites for v in chain])

    def surfaces(self):
        """Eigenvalues of H and of H minus the kinetic energy, in the basis of the bath's
        Schmidt states times the electronic states, and the Schmidt values."""
        A, ne = self.A[0], self.p.n_el
        U, sg, _ = np.linalg.svd(A.reshape(-1, ne), full_matrices=False)
        nb = int((sg > 1e-7).sum())
        B = [np.multiply.outer(U[:, k], np.eye(ne)[l]).reshape(A.shape) for k in range(nb) for l in range(ne)]

        def matrix():
            return np.array([[np.vdot(b, y) for b in B] for y in (self.heff(0, x) for x in B)]).T

        H, keep = matrix(), (self.ops, self.env)
        self.ops, self.env = _operators(self.p, self.t, kinetic=True), {}
        for v in range(self.t.n - 1, 0, -1):
            self.update(v, self.t.parent[v])
        T = matrix()
        self.ops, self.env = keep
        return np.linalg.eigvalsh(H), np.linalg.eigvalsh(H - T), sg[:nb]


def _entropy(r):
    w = np.linalg.eigvalsh(0.5 * (r + r.conj().T))
    w = w[w > 1e-300]
    return float(-(w * np.log(w)).sum())


def _exact_net(case, seed):
    X, Y = _training_set(case, seed)
    x, t = (torch.tensor(a, dtype=torch.float32).double() for a in (X, Y))
    net = surrogate.Net(_widths(case), seed, device="cpu")   # the weights drawn from the seed
    Ws = [w.double().requires_grad_() for w in net.W]
    bs = [b.double().requires_grad_() for b in net.b]
    y = x
    for k, (w, b) in enumerate(zip(Ws, bs)):
        y = y @ w + b
        if k + 1 < len(Ws):
            y = torch.tanh(y)
    if case["kind"] == "infer":
        return dict(y=y.detach())
    (((y - t) ** 2).sum() / (2 * len(x))).backward()
    new = [[(p - 1e-3 * p.grad / (p.grad.abs() + 1e-8)).detach() for p in ps] for ps in (Ws, bs)]  # Adam's first step
    return dict(y=y.detach(), dW=[w.grad for w in Ws], db=[b.grad for b in bs], m=[0.1 * w.grad for w in Ws],
                v=[1e-3 * w.grad ** 2 for w in Ws], W=new[0], b=new[1])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "infer"):
        return _exact_net(case, seed)
    ps = _problems(case, seed)
    if kind == "batch":
        # sweeping some hundred trees in numpy takes minutes
        return None
    flops, _ = _counts(_Tree(ps[0]))
    if case["steps"] * flops > 4e10:
        return None
    s = _Sweep(ps[0])
    s.step(case["dt"], case["steps"])
    bond, occ = s.densities()
    if kind == "step":
        return dict(rho=s.rho(), occ=occ)
    tes, pes, sg = s.surfaces()
    A = s.A[0]
    nn = float(np.linalg.norm(A))
    return dict(rho=s.rho(), norm=nn, energy=float(np.vdot(A, s.heff(0, A)).real) / nn ** 2, occ=occ,
                entropy=np.array([_entropy(s.rho())] + [_entropy(bond[v]) for v in range(1, s.t.n)]),
                tes=tes, pes=pes, sigma=sg)


# ------------------------------------------------------------------ what a pass cannot do without
def _counts(t):
    """(flops of one step, complex values of the state).  A step evolves every tensor twice and
    every bond twice, and moves the centre over every bond four times (one QR, one environment
    update, one absorb each); an exponential takes at least three applications here."""
    flops = size = 0
    for v in range(t.n):
        dims = t.dims(v)
        N = math.prod(dims)
        size += N
        flops += 2 * 3 * 8 * N * sum(dims)
        for u in t.near(v):
            D = dims[t.leg(v, u)]
            # two moves over each bond from either end: QR with Q (16 N D), environment, absorb
            flops += 2 * (16 * N * D + 8 * N * (sum(dims) - D) + 8 * N * D + 8 * N * D)
            flops += 3 * 16 * D ** 3
    return flops, size


def work(case):
    kind = case["kind"]
    if kind in ("train", "infer"):
        w = _widths(case)
        B, par = case["batch"], sum(a * b + b for a, b in zip(w[:-1], w[1:]))
        if kind == "infer":
            return dict(bytes=4.0 * (B * w[0] + par + B * w[-1]), flops=2.0 * B * par)
        # inputs, targets and the output, the gradients, and weights and moments read and written
        return dict(bytes=4.0 * (B * (w[0] + 2 * w[-1]) + 7 * par), flops=6.0 * B * par)
    ts = [_Tree(p) for p in _problems(case, 0)]
    flops, size = (sum(x) for x in zip(*(_counts(t) for t in ts)))
    if kind == "observe":
        # every tensor once down for the densities; the spectra and surfaces are small beside it
        return dict(bytes=16.0 * size, flops=sum(8.0 * math.prod(t.dims(v)) * 2 * sum(t.dims(v)) for t in ts
                                                 for v in range(t.n)))
    return dict(bytes=32.0 * size, flops=float(case["steps"] * flops))
