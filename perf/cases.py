"""Performance cases of the PEPS sampling path: what its users have it do.

A case is one call (or the few calls of one step) through the public Python
entry points, on the lattices, bond dimensions and precisions of the
framework's own workloads: square and rectangular open lattices from 3x3-sized
to 16x16, D from 2 to 10, Dc around 2 D, FP64, FP32 and the mixed path.

Inputs.  Site tensors are a product state plus Gaussian noise of the same
norm, scaled to unit norm per site: their bond spectra decay, as those of
optimised ground states do, so the truncated contraction has a well-defined
value in every precision.  (The i.i.d. tensors of the throughput benchmark
have flat spectra, on which rounding alone moves the result.)  Configurations
are uniform in the S^z = 0 sector.  Everything is drawn from the seed alone.

``exact`` evaluates the same scheme (zip-up with SVD truncation to Dc,
alternating directions, ratios and log-derivatives from the sandwiches of
the configuration's own environments, simple update by QR and SVD) in float64
with plain torch and numpy, batched over the configurations.
"""
import math

import numpy as np
import torch

from paper_1611_09467_gb300 import flops as F
from paper_1611_09467_gb300.peps import PEPS, Packer, SimpleUpdate

J1 = 1.0


def listed():
    return [
        # the plain method on the exactly solvable lattice: one gradient-optimisation step's estimate
        # from 64 configurations; launches and latency count
        dict(name="gradient_4x4_d2_f64", kind="gradient", Lx=4, Ly=4, D=2, Dc=4, J2=0.5, prec="fp64", n=64),
        # the batched plain method: a whole optimisation step's batch at 8x8, D = 4
        dict(name="gradient_8x8_d4_f32", kind="gradient", Lx=8, Ly=8, D=4, Dc=8, J2=0.5, prec="fp32", n=4096),
        # the 10x10 workload in the mixed path, a batch of odd size
        dict(name="gradient_10x10_d6_mixed", kind="gradient", Lx=10, Ly=10, D=6, Dc=12, J2=0.5, prec="mixed_tf32", n=1001),
        # the same model in the FP64 path, which results are checked against
        dict(name="gradient_10x10_d6_f64", kind="gradient", Lx=10, Ly=10, D=6, Dc=12, J2=0.5, prec="fp64", n=76),
        # the headline workload, 16x16 D = 8 Dc = 16 on the tensor cores: the largest case
        dict(name="gradient_16x16_d8_mixed", kind="gradient", Lx=16, Ly=16, D=8, Dc=16, J2=0.5, prec="mixed_tf32", n=1024),
        # the largest bond dimension: psi and E_loc of a few configurations at D = 10, Dc = 20
        dict(name="energy_12x12_d10_f32", kind="energy", Lx=12, Ly=12, D=10, Dc=20, J2=0.5, prec="fp32", n=13),
        # the smallest serving request: psi of one configuration at D = 8, latency alone
        dict(name="amplitude_16x16_d8_f32", kind="amplitudes", Lx=16, Ly=16, D=8, Dc=16, J2=0.5, prec="fp32", n=1),
        # log-derivatives for a natural-gradient step, rectangular lattice, odd D and Dc
        dict(name="derivatives_12x9_d5_f32", kind="derivatives", Lx=12, Ly=9, D=5, Dc=9, J2=0.0, prec="fp32", n=300),
        # sampling: one Metropolis sweep of a batch of chains
        dict(name="sweep_8x8_d4_f64", kind="sweep", Lx=8, Ly=8, D=4, Dc=8, J2=0.5, prec="fp64", n=304),
        # the measured observables: spin correlations of the central 4x4 sites
        dict(name="correlations_6x6_d3_f64", kind="correlations", Lx=6, Ly=6, D=3, Dc=6, J2=0.5, prec="fp64", n=128),
        # the initialiser: Trotter steps of the simple update, next-nearest gates included
        dict(name="simple_update_8x8_d5", kind="simple_update", Lx=8, Ly=8, D=5, Dc=5, J2=0.5, prec="fp64", n=2),
        # serving: small requests of three lattices evaluated together
        dict(name="packed_6_8_10_d4_f32", kind="packed", Lx=6, Ly=6, D=4, Dc=8, J2=0.5, prec="fp32", n=96),
    ]


# ------------------------------------------------------------------ the range
LIMIT_S = 0.7   # a drawn case costs about this at most, by estimate(); the largest listed one costs more


def estimate(c):
    """Rough seconds of one pass, to keep drawn cases within the listed range."""
    D, Dc, sites = c["D"], c["Dc"], c["Lx"] * c["Ly"]
    p, f64 = D * Dc, c["prec"] == "fp64"
    if c["kind"] == "simple_update":
        return c["n"] * (22 if c["J2"] else 4) * (4e-4 + 6e-6 * D ** 4)
    # a boundary sweep's absorption of one site with its cut, and the sandwiches of one site
    cut = (5e-5 + 1.8e-5 * p if f64 else 3e-5 + 2.6e-6 * p) if p <= 128 else (1.2e-2 if f64 else 8e-3) * (p / 200.0) ** 2
    tuned = Dc == 2 * D and D in (2, 4, 6, 8) and not (f64 and D > 4)
    step = (2e-5 + 7.0 * Dc * Dc * D ** 5 / (1.5e9 if f64 else 8e9)) * (1.0 if tuned else 3.0)
    per = {"amplitudes": cut, "derivatives": 2 * cut + step / D, "energy": 2 * cut + step, "gradient": 2 * cut + step,
           "packed": 8 * cut + 8 * step, "sweep": 8 * cut + 4 * step, "correlations": (10 if f64 else 6) * cut}[c["kind"]]
    side = 450.0 if p <= 72 else 300.0     # sweeps that run side by side
    return sites * per * max(1.0, c["n"] / side)


def draw(rng):
    while True:
        kind = rng.choice(["gradient"] * 4 + ["energy", "energy", "amplitudes", "amplitudes", "derivatives",
                                             "derivatives", "sweep", "correlations", "simple_update", "packed"])
        D = int(round(math.exp(rng.uniform(math.log(2), math.log(10.4)))))
        Dc = 2 * D if rng.random() < 0.6 else rng.randint(D, min(32, 256 // D, 3 * D))
        Lx = int(round(math.exp(rng.uniform(math.log(3), math.log(16)))))
        Ly = int(round(math.exp(rng.uniform(math.log(3), math.log(16)))))
        if Lx * Ly % 2:
            continue
        c = dict(kind=kind, Lx=Lx, Ly=Ly, D=D, Dc=Dc, J2=rng.choice([0.0, 0.5, 0.5]),
                 prec=rng.choice(["fp64", "fp32", "mixed_tf32"]), n=int(round(math.exp(rng.uniform(0.0, math.log(4096))))))
        if kind == "simple_update":
            c.update(prec="fp64", Dc=D, D=min(D, 6), n=rng.randint(1, 4))
            c["Dc"] = c["D"]
        if kind == "correlations":
            c["n"] = min(c["n"], 512)
        if kind == "packed":
            c["n"] = max(c["n"], 4)
        while c["n"] > 1 and estimate(c) > LIMIT_S:
            c["n"] = c["n"] * 3 // 4
        if kind == "packed" and c["n"] < 4:
            continue
        if estimate(c) <= LIMIT_S:
            return c


# -------------------------------------------------------------------- inputs
def _tensors(Lx, Ly, D, seed):
    """[N][2][D][D][D][D] float64 on the GPU: product state plus noise, unit norm per site, open edges."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    N = Lx * Ly
    A = torch.randn((N, 2, D, D, D, D), dtype=torch.float64, device="cuda", generator=g) / math.sqrt(2 * D ** 4)
    t = math.pi / 8 + math.pi / 4 * torch.rand(N, dtype=torch.float64, device="cuda", generator=g)
    A[:, 0, 0, 0, 0, 0] += torch.cos(t)
    A[:, 1, 0, 0, 0, 0] += torch.sin(t)
    V = A.view(Ly, Lx, 2, D, D, D, D)
    V[:, 0, :, 1:] = 0
    V[:, -1, :, :, 1:] = 0
    V[0, :, :, :, :, 1:] = 0
    V[-1, :, :, :, :, :, 1:] = 0
    return A / A.flatten(1).norm(dim=1).view(-1, 1, 1, 1, 1, 1)


def _spins(n, N, seed):
    """[n][N] uniformly random S^z = 0 configurations (0 / 1) on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed + 7919)
    r = torch.rand((n, N), dtype=torch.float64, device="cuda", generator=g)
    s = torch.zeros((n, N), dtype=torch.int64, device="cuda")
    return s.scatter_(1, r.argsort(dim=1)[:, : N // 2], 1)


def _pack(s):
    n, N = s.shape
    words = -(-N // 64)
    s = torch.nn.functional.pad(s, (0, words * 64 - N)).view(n, words, 64)
    return (s << torch.arange(64, device=s.device)).sum(2).contiguous()


def _centre(c):
    """The central sites that correlations are measured on: up to 4 x 4."""
    w, h = min(4, c["Lx"]), min(4, c["Ly"])
    x0, y0 = (c["Lx"] - w) // 2, (c["Ly"] - h) // 2
    return [(y0 + y) * c["Lx"] + x0 + x for y in range(h) for x in range(w)]


def _requests(c):
    """(Lx, Ly, n) of the requests of a packed case: growing lattices, shrinking batches."""
    return [(c["Lx"] + 2 * k, c["Ly"] + 2 * k, c["n"] // (k + 1)) for k in range(3)]


def _start_state(c, seed):
    """Gamma and bond weights a simple-update run starts from: random tensors, slowly decaying weights."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    Lx, Ly, D = c["Lx"], c["Ly"], c["D"]
    G = torch.randn((Lx * Ly, 2, D, D, D, D), dtype=torch.float64, device="cuda", generator=g)
    V = G.view(Ly, Lx, 2, D, D, D, D)
    V[:, 0, :, 1:] = 0
    V[:, -1, :, :, 1:] = 0
    V[0, :, :, :, :, 1:] = 0
    V[-1, :, :, :, :, :, 1:] = 0
    G = G / G.flatten(1).norm(dim=1).view(-1, 1, 1, 1, 1, 1)
    lam = 0.7 ** torch.arange(D, dtype=torch.float64, device="cuda")
    lam = (lam / lam.norm()).repeat(Ly * (Lx - 1) + (Ly - 1) * Lx, 1)
    return G, lam


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "simple_update":
        G, lam = _start_state(c, seed)
        su = SimpleUpdate(G.cpu().numpy(), lam.cpu().numpy(), c["Lx"], c["Ly"], c["D"], J1=J1, J2=c["J2"])
        return dict(case=c, su=su, G=su.Gam.clone(), lam=su.lam.clone())
    if kind == "packed":
        reqs = []
        for k, (Lx, Ly, n) in enumerate(_requests(c)):
            A = _tensors(Lx, Ly, c["D"], seed + 101 * k)
            m = PEPS(A.cpu().numpy(), Lx, Ly, c["D"], c["Dc"], J1=J1, J2=c["J2"], prec=c["prec"])
            reqs.append((m, _pack(_spins(n, Lx * Ly, seed + 101 * k))))
        return dict(case=c, packer=Packer(), reqs=reqs)
    A = _tensors(c["Lx"], c["Ly"], c["D"], seed)
    m = PEPS(A.cpu().numpy(), c["Lx"], c["Ly"], c["D"], c["Dc"], J1=J1, J2=c["J2"], prec=c["prec"])
    return dict(case=c, m=m, S=_pack(_spins(c["n"], c["Lx"] * c["Ly"], seed)), seed=seed, sites=_centre(c))


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "simple_update":
        su = state["su"]
        su.Gam.copy_(state["G"])           # every pass starts from the same tensors
        su.lam.copy_(state["lam"])
        change = su.evolve(0.01, c["n"])
        return dict(A=su.to_peps(), Gam=su.Gam, lam=su.lam, change=change)
    if kind == "packed":
        return state["packer"].evaluate(state["reqs"], eloc=True)
    m, S = state["m"], state["S"]
    if kind == "gradient":
        return m.gradient(S, per_config=True)
    if kind == "energy":
        return m.evaluate(S, logabs=True, eloc=True)
    if kind == "amplitudes":
        logabs, sign, status = m.amplitudes(S)
        return dict(logabs=logabs, sign=sign, status=status)
    if kind == "derivatives":
        return m.log_derivatives(S)
    if kind == "sweep":
        S = S.clone()                      # the chains move in place; every pass starts from the same ones
        return dict(accepted=m.mc_sweep(S, 1, seed=state["seed"]), S=S)
    return m.correlations(S, state["sites"])


# ---------------------------------------------------------------------- work
def _sample_spins(Lx, Ly):
    r = np.random.RandomState(1).rand(4, Lx * Ly)
    return (r.argsort(1).argsort(1) < Lx * Ly // 2).astype(np.int64)


def work(case):
    return {k: float(v) for k, v in _work(case).items()}


def _work(case):
    c, kind = case, case["kind"]
    Lx, Ly, D, Dc, n = c["Lx"], c["Ly"], c["D"], c["Dc"], c["n"]
    wide = 8 if c["prec"] == "fp64" else 4
    A_bytes = 2 * Lx * Ly * D ** 4 * wide
    if kind == "simple_update":
        bonds = Ly * (Lx - 1) + (Ly - 1) * Lx
        if c["J2"]:
            bonds += 6 * (Ly - 1) * (Lx - 1)
        # two thin QRs and their application to D columns, the reduced SVD
        per = 2 * (2 * D ** 3 * (2 * D) ** 2 + 4 * D ** 3 * 2 * D * 2 * D) + 20 * (4 * D) ** 3
        return dict(bytes=float(2 * 8 * 2 * Lx * Ly * D ** 4 * 2), flops=float(n * bonds * per))
    if kind == "packed":
        got = [_work(dict(c, kind="energy", Lx=x, Ly=y, n=k)) for x, y, k in _requests(c)]
        return {k: sum(w[k] for w in got) for k in ("bytes", "flops")}
    W, spins = F.Work(Lx, Ly, D, Dc), _sample_spins(Lx, Ly)
    boundary = F.boundary_flops(Lx, Ly, D, Dc)
    row = lambda O: float(np.mean([W.row_flops(s, O) for s in spins]))  # noqa: E731
    pair = lambda J2: float(np.mean([W.pair_flops(s, J2) for s in spins]))  # noqa: E731
    S_bytes = n * -(-Lx * Ly // 64) * 8
    if kind == "gradient":
        return dict(bytes=float(A_bytes + S_bytes + 2 * 2 * Lx * Ly * D ** 4 * 8 + n * 21),
                    flops=n * (boundary + row(True) + pair(c["J2"]) + 4.0 * Lx * Ly * D ** 4))
    if kind == "energy":
        return dict(bytes=float(A_bytes + S_bytes + n * 21), flops=n * (boundary + row(False) + pair(c["J2"])))
    if kind == "amplitudes":
        return dict(bytes=float(A_bytes + S_bytes + n * 13), flops=n * boundary * Ly / (2.0 * Ly - 1))
    if kind == "derivatives":
        return dict(bytes=float(A_bytes + S_bytes + n * Lx * Ly * D ** 4 * wide), flops=n * (boundary + W.row_flops(None, True)))
    if kind == "sweep":
        return dict(bytes=float(A_bytes + 2 * S_bytes + 8 * n), flops=n * (2 * boundary + row(False) + pair(0.0)))
    nc = len(_centre(c))
    rows_below = sum(Ly - 1 - i // Lx for i in _centre(c))
    return dict(bytes=float(A_bytes + S_bytes + n * 12 + nc * nc * 8),
                flops=n * (boundary + row(False) + rows_below * boundary / (2.0 * Ly - 1) + (rows_below + nc) * row(True) / Ly))


# --------------------------------------------------- the scheme in 64 bits
E = torch.einsum


def _svd(X):
    """Batched float64 SVD: on the GPU where its batched solver applies, else on the host."""
    if max(X.shape[-2:]) <= 32:
        return torch.linalg.svd(X, full_matrices=False)
    U, s, V = torch.linalg.svd(X.cpu(), full_matrices=False)
    return U.to(X.device), s.to(X.device), V.to(X.device)


def _absorb(mps, row, Dc, rightward):
    """One row ([n][l][r][in][out] per column) into the boundary MPS ([n][a][p][b]); the new MPS and ln of its norm."""
    L, n = len(row), row[0].shape[0]
    C = torch.ones((n, 1, 1, 1), dtype=torch.float64, device=row[0].device)
    out = [None] * L
    for step in range(L):
        c = step if rightward else L - 1 - step
        if rightward:
            X = E("nklpb,nlrpo->nkobr", E("nkal,napb->nklpb", C, mps[c]), row[c])
        else:
            X = E("nkrpa,nlrpo->nkoal", E("nkbr,napb->nkrpa", C, mps[c]), row[c])
        _, k, o, a, l = X.shape
        if step == L - 1:
            T = X.reshape(n, k, o, a * l)
            norm = T.flatten(1).norm(dim=1)
            T = T / norm.view(-1, 1, 1, 1)
            out[c] = T if rightward else T.permute(0, 3, 2, 1)
            return out, norm.log()
        M = X.reshape(n, k * o, a * l)
        K = min(Dc, k * o, a * l)
        U = _svd(M)[0][:, :, :K]
        out[c] = U.reshape(n, k, o, K) if rightward else U.reshape(n, k, o, K).permute(0, 3, 2, 1)
        C = (U.transpose(1, 2) @ M).reshape(n, K, a, l)


class _Scheme:
    """Environments and sandwiches of a batch of configurations ([n][N] spins)."""

    def __init__(self, A, s, Lx, Ly, Dc, both=True):
        self.A, self.s, self.Lx, self.Ly, self.Dc = A, s, Lx, Ly, Dc
        self.n, self.D = s.shape[0], A.shape[2]
        self.T = [self.pick(i, s[:, i]) for i in range(Lx * Ly)]
        one = [torch.ones((self.n, 1, 1, 1), dtype=torch.float64, device=A.device)] * Lx
        self.up, self.ln = [one], [torch.zeros(self.n, dtype=torch.float64, device=A.device)]
        for r in range(Ly):
            m, ln = _absorb(self.up[-1], self.row(r), Dc, r % 2 == 0)
            self.up.append(m)
            self.ln.append(self.ln[-1] + ln)
        v = torch.ones((self.n, 1), dtype=torch.float64, device=A.device)
        for M in self.up[Ly]:
            v = E("na,nab->nb", v, M[:, :, 0])
        self.logabs = self.ln[Ly] + v[:, 0].abs().log()
        if both:
            self.dn = [None] * Ly + [one]
            for r in range(Ly - 1, 0, -1):
                flipped = [t.transpose(3, 4) for t in self.row(r)]
                self.dn[r] = _absorb(self.dn[r + 1], flipped, Dc, (Ly - 1 - r) % 2 == 0)[0]

    def pick(self, i, spin):
        """[n][l][r][u][d] of site i at the given spins, cut to the true bonds."""
        r, c, D = i // self.Lx, i % self.Lx, self.D
        l, rr = 1 if c == 0 else D, 1 if c == self.Lx - 1 else D
        u, d = 1 if r == 0 else D, 1 if r == self.Ly - 1 else D
        return self.A[i, :, :l, :rr, :u, :d][spin]

    def row(self, r):
        return self.T[r * self.Lx:(r + 1) * self.Lx]

    def flip(self, i):
        return self.pick(i, 1 - self.s[:, i])

    @staticmethod
    def left1(X, u, T, d):
        return E("nbqrd,nqdc->nbrc", E("nqblu,nlrud->nbqrd", E("nalq,naub->nqblu", X, u), T), d)

    @staticmethod
    def right1(X, u, T, d):
        return E("naqld,npdq->nalp", E("nauqr,nlrud->naqld", E("naub,nbrq->nauqr", u, X), T), d)

    @staticmethod
    def left2(X, u, T, V, d):
        P = E("nalmq,naub->nlmqub", X, u)
        P = E("nlmqub,nlrux->nmqbrx", P, T)
        P = E("nmqbrx,nmsxd->nqbrsd", P, V)
        return E("nqbrsd,nqdc->nbrsc", P, d)

    @staticmethod
    def right2(X, u, T, V, d):
        P = E("naub,nbrsc->naursc", u, X)
        P = E("naursc,nlrux->nascxl", P, T)
        P = E("nascxl,nmsxd->nacldm", P, V)
        return E("nacldm,nqdc->nalmq", P, d)

    def one(self, k):
        return torch.ones((self.n,) + (1,) * k, dtype=torch.float64, device=self.A.device)

    def single_rows(self, energy, derivs):
        """Sum of J1/2 ratios of horizontal exchanges, and the log-derivatives [n][N][D^4]."""
        Lx, s, e = self.Lx, self.s, 0.0
        N, D = Lx * self.Ly, self.D
        O = torch.zeros((self.n, N, D, D, D, D), dtype=torch.float64, device=self.A.device) if derivs else None
        for r in range(self.Ly):
            u, d, T = self.up[r], self.dn[r + 1], self.row(r)
            G = [None] * Lx + [self.one(3)]
            for c in range(Lx - 1, -1, -1):
                G[c] = self.right1(G[c + 1], u[c], T[c], d[c])
            W, X = G[0].reshape(self.n), self.one(3)
            for c in range(Lx):
                i = r * Lx + c
                if derivs:
                    P = E("nalq,naub->nlqub", X, u[c])
                    Q = E("nqdc,nbrc->nqdbr", d[c], G[c + 1])
                    B = E("nlqub,nqdbr->nlrud", P, Q) / W.view(-1, 1, 1, 1, 1)
                    O[:, i, :B.shape[1], :B.shape[2], :B.shape[3], :B.shape[4]] = B
                if c + 1 < Lx:
                    if energy:
                        Y = self.left1(X, u[c], self.flip(i), d[c])
                        Y = self.left1(Y, u[c + 1], self.flip(i + 1), d[c + 1])
                        w = (Y * G[c + 2]).flatten(1).sum(1) / W
                        e = e + 0.5 * J1 * torch.where(s[:, i] != s[:, i + 1], w, 0.0)
                    X = self.left1(X, u[c], T[c], d[c])
        return e, None if O is None else O.view(self.n, N, D ** 4)

    def row_pairs(self, J2):
        """Sum of J/2 ratios of vertical and diagonal exchanges."""
        Lx, s, e = self.Lx, self.s, 0.0
        for r in range(self.Ly - 1):
            u, d, T, V = self.up[r], self.dn[r + 2], self.row(r), self.row(r + 1)
            H = [None] * Lx + [self.one(4)]
            for c in range(Lx - 1, -1, -1):
                H[c] = self.right2(H[c + 1], u[c], T[c], V[c], d[c])
            W, X = H[0].reshape(self.n), self.one(4)
            for c in range(Lx):
                i, j = r * Lx + c, (r + 1) * Lx + c
                Y = self.left2(X, u[c], self.flip(i), self.flip(j), d[c])
                w = (Y * H[c + 1]).flatten(1).sum(1) / W
                e = e + 0.5 * J1 * torch.where(s[:, i] != s[:, j], w, 0.0)
                if c + 1 == Lx:
                    break
                if J2:
                    for a, b in ((i, j + 1), (i + 1, j)):
                        t = {k: self.T[k] for k in (i, j, i + 1, j + 1)}
                        t[a], t[b] = self.flip(a), self.flip(b)
                        Y = self.left2(X, u[c], t[i], t[j], d[c])
                        Y = self.left2(Y, u[c + 1], t[i + 1], t[j + 1], d[c + 1])
                        w = (Y * H[c + 2]).flatten(1).sum(1) / W
                        e = e + 0.5 * J2 * torch.where(s[:, a] != s[:, b], w, 0.0)
                X = self.left2(X, u[c], T[c], V[c], d[c])
        return e

    def diagonal(self, J2):
        z = 0.5 - self.s.view(self.n, self.Ly, self.Lx).double()
        e = J1 * ((z[:, :, 1:] * z[:, :, :-1]).sum((1, 2)) + (z[:, 1:] * z[:, :-1]).sum((1, 2)))
        return e + J2 * ((z[:, 1:, 1:] * z[:, :-1, :-1]).sum((1, 2)) + (z[:, 1:, :-1] * z[:, :-1, 1:]).sum((1, 2)))

    def sandwich(self, u, T, d):
        X = self.one(3)
        for c in range(self.Lx):
            X = self.left1(X, u[c], T[c], d[c])
        return X.reshape(self.n)

    def correlations(self, sites):
        """(m2 [n], sums [nc][nc]) of the local S_p.S_q on the given sites."""
        Lx, Ly, n, nc = self.Lx, self.Ly, self.n, len(sites)
        z = 0.5 - self.s.double()
        W = {r: self.sandwich(self.up[r], self.row(r), self.dn[r + 1]) for r in {i // Lx for i in sites}}
        local = torch.zeros((n, nc, nc), dtype=torch.float64, device=self.A.device)
        for p, i in enumerate(sites):
            local[:, p, p] = 0.75
            ri = i // Lx
            u, ln, T = self.up[ri], self.ln[ri], list(self.row(ri))
            T[i % Lx] = self.flip(i)
            for r in range(ri, Ly):
                for q, j in enumerate(sites):
                    if j <= i or j // Lx != r:
                        continue
                    V = list(T)
                    V[j % Lx] = self.flip(j)
                    w = self.sandwich(u, V, self.dn[r + 1]) / W[r] * (ln - self.ln[r]).exp()
                    v = z[:, i] * z[:, j] + torch.where(self.s[:, i] != self.s[:, j], 0.5 * w, 0.0)
                    local[:, p, q] = local[:, q, p] = v
                if r + 1 < Ly:
                    u, more = _absorb(u, T, self.Dc, r % 2 == 0)
                    ln, T = ln + more, list(self.row(r + 1))
        eps = torch.tensor([(-1.0) ** (i // Lx + i % Lx) for i in sites], dtype=torch.float64, device=local.device)
        return E("npq,p,q->n", local, eps, eps) / nc ** 2, local.sum(0)


def _su_exact(c, seed):
    """Bond weights and the change of the last step after the case's Trotter steps."""
    Lx, Ly, D, J2, dtau = c["Lx"], c["Ly"], c["D"], c["J2"], 0.01
    G, lam = (t.cpu().numpy().copy() for t in _start_state(c, seed))
    nh = Ly * (Lx - 1)

    def bond(i, leg):
        r, x = divmod(i, Lx)
        return [r * (Lx - 1) + x - 1 if x else -1, r * (Lx - 1) + x if x < Lx - 1 else -1,
                nh + (r - 1) * Lx + x if r else -1, nh + r * Lx + x if r < Ly - 1 else -1][leg]

    def weight(t, i, legs, f):
        for leg in legs:
            b = bond(i, leg)
            if b >= 0:
                t = t * f(lam[b]).reshape([1] + [D if k == leg else 1 for k in range(4)])
        return t

    def inv(w):
        return np.where(w != 0, 1 / np.where(w != 0, w, 1), 0.0)

    def gate(J):
        ps = np.zeros((4, 4))
        ps[1:3, 1:3] = [[0.5, -0.5], [-0.5, 0.5]]
        return math.exp(-dtau * J / 4) * (np.eye(4) - ps) + math.exp(0.75 * dtau * J) * ps

    swap = np.eye(4)[[0, 2, 1, 3]]

    def apply(i, j, g):
        li, lj = (1, 0) if j == i + 1 else (3, 2)
        b = bond(i, li)
        A = weight(weight(G[i], i, [k for k in range(4) if k != li], lambda w: w), i, [li], lambda w: w)
        B = weight(G[j], j, [k for k in range(4) if k != lj], lambda w: w)
        A, B = np.moveaxis(A, [0, 1 + li], [3, 4]), np.moveaxis(B, [0, 1 + lj], [3, 4])     # [outer][s][x]
        Qi, Ri = np.linalg.qr(A.reshape(D ** 3, 2 * D))
        Qj, Rj = np.linalg.qr(B.reshape(D ** 3, 2 * D))
        ki, kj = Ri.shape[0], Rj.shape[0]
        th = np.einsum("asx,btx->asbt", Ri.reshape(ki, 2, D), Rj.reshape(kj, 2, D))
        th = np.einsum("pqst,asbt->apqb", g.reshape(2, 2, 2, 2), th)
        U, sv, Vt = np.linalg.svd(th.reshape(2 * ki, 2 * kj), full_matrices=False)
        K = min(D, len(sv))
        lam[b] = 0
        lam[b][:K] = sv[:K] / np.linalg.norm(sv[:K])
        Ni, Nj = np.zeros((D ** 3, 2, D)), np.zeros((D ** 3, 2, D))
        Ni[:, :, :K] = np.einsum("ra,asx->rsx", Qi, U[:, :K].reshape(ki, 2, K))
        Nj[:, :, :K] = np.einsum("rb,xsb->rsx", Qj, Vt[:K].reshape(K, 2, kj))
        for site, leg, N in ((i, li, Ni), (j, lj, Nj)):
            t = np.moveaxis(N.reshape(D, D, D, 2, D), [3, 4], [0, 1 + leg])
            t = weight(t, site, [k for k in range(4) if k != leg], inv)
            r, x = divmod(site, Lx)
            for k, edge in enumerate((x == 0, x == Lx - 1, r == 0, r == Ly - 1)):
                if edge:
                    t = np.moveaxis(np.moveaxis(t, 1 + k, 0) * (np.arange(D) == 0).reshape(-1, 1, 1, 1, 1), 0, 1 + k)
            G[site] = t

    def tensors():
        A = np.stack([weight(G[i], i, range(4), np.sqrt) for i in range(Lx * Ly)])
        return A / np.sqrt((A ** 2).sum(axis=(1, 2, 3, 4, 5), keepdims=True))

    for step in range(c["n"]):
        for par in (0, 1):
            for r in range(Ly):
                for x in range(par, Lx - 1, 2):
                    apply(r * Lx + x, r * Lx + x + 1, gate(J1))
        for par in (0, 1):
            for r in range(par, Ly - 1, 2):
                for x in range(Lx):
                    apply(r * Lx + x, (r + 1) * Lx + x, gate(J1))
        if J2:
            for kind in (0, 1):
                for cp in (0, 1):
                    for rp in (0, 1):
                        at = [r * Lx + x for r in range(rp, Ly - 1, 2) for x in range(cp, Lx - 1, 2)]
                        for sub in range(3):
                            for a in at:
                                m, k = (a + 1, a + 1 + Lx) if kind == 0 else (a, a + Lx)
                                if sub == 1:
                                    apply(min(m, k), max(m, k), gate(J2))
                                else:
                                    apply(a, a + 1, swap)
    # Gamma, A and the change of a step depend on the singular vectors' signs
    return dict(A=None, Gam=None, lam=torch.from_numpy(lam), change=None)


def _exact_seconds(c):
    """Rough seconds of exact(): its SVDs and contractions."""
    if c["kind"] == "simple_update":
        return c["n"] * c["Lx"] * c["Ly"] * (14 if c["J2"] else 2) * (4e-4 + 1.2e-8 * c["D"] ** 6)
    p = c["D"] * c["Dc"]
    svd = 2e-5 if p <= 32 else 1e-4 + 4e-9 * p ** 3
    per = 2 * c["Lx"] * c["Ly"] * svd
    if c["kind"] == "correlations":
        per *= 1 + len(_centre(c)) / 4
    if c["kind"] in ("gradient", "energy", "packed"):
        per += c["Lx"] * c["Ly"] * 40 * c["Dc"] ** 2 * c["D"] ** 5 / 3e11
    return c["n"] * per * (6 if c["kind"] == "packed" else 1)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "sweep" or _exact_seconds(c) > 13:      # a sweep returns whole numbers
        return None
    if kind == "simple_update":
        return _su_exact(c, seed)
    if kind == "packed":
        out = []
        for k, (Lx, Ly, n) in enumerate(_requests(c)):
            q = _energies(dict(c, Lx=Lx, Ly=Ly, n=n), seed + 101 * k)
            out.append(dict(logabs=q.logabs, sign=None, eloc=q.eloc, O=None, status=None))
        return out
    if kind in ("gradient", "energy"):
        q = _energies(c, seed, derivs=kind == "gradient")
        if kind == "energy":
            return dict(logabs=q.logabs, sign=None, eloc=q.eloc, O=None, status=None)
        N, D4, n = c["Lx"] * c["Ly"], c["D"] ** 4, c["n"]
        up = (q.s == 0).double()
        cov = torch.empty((N, 2, D4), dtype=torch.float64, device=q.s.device)
        for sp, sel in ((0, up), (1, 1 - up)):
            mean = E("ni,nix->ix", sel, q.O) / n
            cov[:, sp] = E("n,ni,nix->ix", q.eloc, sel, q.O) / n - q.eloc.mean() * mean
        return dict(energy_per_site=float(q.eloc.mean()) / N, grad=2 * cov, cov=cov, n_used=None, logabs=q.logabs,
                    sign=None, eloc=q.eloc, status=None)
    q = _Scheme(_tensors(c["Lx"], c["Ly"], c["D"], seed), _spins(c["n"], c["Lx"] * c["Ly"], seed), c["Lx"], c["Ly"],
                c["Dc"], both=kind != "amplitudes")
    if kind == "amplitudes":
        return dict(logabs=q.logabs, sign=None, status=None)
    if kind == "derivatives":
        return q.single_rows(False, True)[1]
    m2, corr = q.correlations(_centre(c))
    return dict(m2=m2, corr=corr, status=None)


def _energies(c, seed, derivs=False):
    q = _Scheme(_tensors(c["Lx"], c["Ly"], c["D"], seed), _spins(c["n"], c["Lx"] * c["Ly"], seed), c["Lx"], c["Ly"],
                c["Dc"])
    h, q.O = q.single_rows(True, derivs)
    q.eloc = h + q.row_pairs(c["J2"]) + q.diagonal(c["J2"])
    return q
