"""Performance cases of the superposition-of-Gaussian-states library: the calls a user's program makes,
over the sizes, ranks and precisions the repository's workloads span.

A case names one call of ``paper_2105_01088_gb300.Solver`` on a problem of given size:

  step        continue a solve from host states: set_state, step(steps), get_state
  serve       the same for several uneven problems live in one solver (continuous batching), one step
              of all of them per call
  energy      the energy and the pair matrices (G, h) of the current states
  correlator  <S(0).S(r)> on every site, or K(r) of the two-channel Kondo model
  variance    <H> and <H^2> - <H>^2
  renyi       the Renyi-2 entropy of growing subsystems

``model``: "anderson" (``bath`` sites per channel, ``channels``) or "kondo" (two channels, ``length``); the
matrix size is 4 x the number of sites.  States are drawn as a grown ansatz has them: rotations exp(K) of one
random pure state, with overlaps of order one.
"""
import itertools
import math

import numpy as np
import torch

import paper_2105_01088_gb300 as sgs

PRECISIONS = {"fp64": sgs.SGS_FP64, "tf32": sgs.SGS_MIXED_TF32, "bf16": sgs.SGS_MIXED_BF16,
              "3xtf32": sgs.SGS_FP32_3XTF32}


def _case(name, call, bath, rank, **more):
    c = {"name": name, "call": call, "model": "anderson", "bath": bath, "channels": 1, "rank": rank, "steps": 1,
         "precision": "fp64", "phase_c": False, "parity": 1, "dtau": 0.05, "U": 4.0, "V": 0.5, "scratch_gb": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest configured workload (16 sites, 4 states): a chain of short launches
        _case("step_L16_M4", "step", 15, 4, U=2.0, steps=4),
        # a serving iteration: eight live solves of 9 to 41 sites and 4 or 8 states, TF32 equation of motion
        _case("serve_8x_L9-41", "serve", 40, 8, slots=8, bath_min=8, precision="tf32", phase_c=True),
        # (E, G, h) of a mid-sized ansatz: the forward part of a step on its own
        _case("energy_L41_M6", "energy", 40, 6),
        # an instance of the batched distribution, ordinary size (61 sites, 16 states)
        _case("step_L61_M16", "step", 60, 16, phase_c=True),
        # the benchmark workload, in both of its precisions, with the benchmark's slice scratch
        _case("step_L128_M32", "step", 127, 32, scratch_gb=6.0),
        _case("step_L128_M32_tf32", "step", 127, 32, precision="tf32", scratch_gb=6.0),
        # the paper's largest system (Sec. IV A) at the rank the repository's growth run reaches
        _case("step_L500_M8", "step", 499, 8, U=1.0, V=0.2 ** 0.5, dtau=0.1, phase_c=True),
        # the two-channel impurity's system in the precision it is run in, rank as grown so far
        _case("step_2ch_L201_M16_3xtf32", "step", 100, 16, channels=2, U=8.0, V=0.6, parity=-1, precision="3xtf32"),
        # observables after a solve: screening cloud K(r) of the two-channel Kondo lattice
        _case("kondo_K_L20_M8", "correlator", 0, 8, model="kondo", length=20, J=1.0, t=0.5),
        # the point of the energy extrapolation
        _case("variance_L97_M10", "variance", 96, 10),
        # entropies of the impurity with 2, 7 and 12 sites, and of a block beyond shared memory
        _case("renyi_L41_M6", "renyi", 40, 6, blocks=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["step", "step", "step", "step", "serve", "energy", "correlator", "variance", "renyi"])
    U, V = round(rng.uniform(0.5, 8.0), 3), round(rng.uniform(0.2, 1.0), 3)
    phase = rng.random() < 0.5
    if call == "serve":
        lo = rng.randint(8, 16)
        return _case("", call, rng.randint(24, 40), 8, slots=rng.randint(3, 8), bath_min=lo, U=U, V=V, phase_c=True,
                     precision=rng.choice(["tf32", "fp64"]))
    if call == "renyi":
        return _case("", call, rng.randint(17, 48), rng.randint(3, 6), U=U, V=V, blocks=rng.randint(2, 4))
    if call == "correlator" and rng.random() < 0.5:
        return _case("", call, 0, rng.randint(3, 10), model="kondo", length=rng.randint(6, 30),
                     J=round(rng.uniform(0.2, 2.0), 3), t=0.5)
    channels = 2 if call == "step" and rng.random() < 0.2 else 1
    bath = _log_int(rng, 12, 499 if call == "step" else 140) // channels
    n = 4 * (1 + channels * bath)
    # ranks up to 32, with no more pair work than the benchmark's, and pair buffers within some tens of GB
    most = 32
    while most > 4 and most * (most - 1) / 2 * n ** 3 > 6.7e10:
        most -= 1
    rank = _log_int(rng, 3, most)
    prec = rng.choice(["fp64", "fp64", "tf32", "3xtf32"]) if call == "step" else "fp64"
    return _case("", call, bath, rank, channels=channels, U=U, V=V, phase_c=phase, precision=prec,
                 steps=rng.choice([1, 2, 4]) if call == "step" and n < 160 else 1)


# ------------------------------------------------------------------ sizes

def _problems(case):
    """[(bath sites per channel, rank)] of the case's live problems."""
    if case["call"] != "serve":
        return [(case["bath"], case["rank"])]
    k, lo, hi = case["slots"], case["bath_min"], case["bath"]
    return [(lo + (hi - lo) * i // max(k - 1, 1), case["rank"] if i % 2 else max(case["rank"] // 2, 1))
            for i in range(k)]


def _n(case, bath):
    return 8 * case["length"] if case["model"] == "kondo" else 4 * (1 + case["channels"] * bath)


def _blocks(case):
    """Chain sites beside the impurity of each Renyi subsystem."""
    return [2, 7, 12, 16][:case["blocks"]]


def work(case):
    flops = bytes_ = 0.0
    for bath, M in _problems(case):
        n, P = _n(case, bath), M * (M - 1) / 2
        n3 = float(n) ** 3
        pairs = (2.0 + 1.0) * n3 * P + 4.0 / 3.0 * n3 * max(P - (M - 1), 0)     # inverse, Im Delta, Pfaffian
        if case["call"] in ("step", "serve"):
            flops += case["steps"] * (pairs + 4.0 * n3 * P + 16.0 * n3 * M)     # W, V, X; the states' update
            bytes_ += 2.0 * 8.0 * M * n * n
        else:
            flops += pairs
            bytes_ += 8.0 * M * n * n
            if case["call"] == "renyi":
                for l in _blocks(case):
                    flops += M * M * (M * M + 1) / 2 * 4.0 / 3.0 * (8.0 * (1 + l)) ** 3
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _states(n, M, seed, parity, spread=1.0):
    """[M, n, n] pure covariance matrices: rotations exp(K_mu) of one Haar-random state of the given parity."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device=dev, dtype=torch.float64)

    Q, R = torch.linalg.qr(normal(n, n))
    Q = Q * torch.sign(torch.diagonal(R))
    if torch.linalg.slogdet(Q)[0].item() * parity < 0:
        Q[:, 0] = -Q[:, 0]
    base = Q[:, 0::2] @ Q[:, 1::2].T
    base = base - base.T
    out = []
    for _ in range(M):
        K = normal(n, n) * (spread / n)
        O = torch.linalg.matrix_exp(K - K.T)
        G = O @ base @ O.T
        out.append(0.5 * (G - G.T))
    return torch.stack(out)


def _model(case, bath):
    if case["model"] == "kondo":
        return sgs.build_2ck(case["length"], case["J"], case["t"])
    return sgs.build_anderson(bath, case["U"], -case["U"] / 2, case["V"], n_channels=case["channels"])


def _pinned(shape):
    t = torch.empty(shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    return t.numpy()


def prepare(case, seed):
    sgs.use_torch_allocator()
    models, hosts = [], []
    for i, (bath, M) in enumerate(_problems(case)):
        models.append(_model(case, bath))
        g = _pinned((M, models[-1].n, models[-1].n))
        g[...] = _states(models[-1].n, M, seed * 64 + i, case["parity"]).cpu().numpy()
        hosts.append(g)
    solver = sgs.Solver(models, hosts, None, dtau=case["dtau"], precision=PRECISIONS[case["precision"]],
                        cmode=sgs.SGS_C_PHASE if case["phase_c"] else sgs.SGS_C_INVERSE, parity=case["parity"],
                        emulation_scratch=int(case["scratch_gb"] * 1e9))
    return {"case": case, "solver": solver, "hosts": hosts, "out": [_pinned(g.shape) for g in hosts]}


def run(state):
    case, s = state["case"], state["solver"]
    call = case["call"]
    if call in ("step", "serve"):
        for i, g in enumerate(state["hosts"]):
            s.set_state(g, instance=i)
        E = s.step(case["steps"])
        got = {"energies": E}
        for i, buf in enumerate(state["out"]):
            gamma, lam = s.get_state(i, out=buf)
            got[f"gamma{i}"], got[f"lambda{i}"] = gamma, lam
        return got
    if call == "energy":
        E = s.energy()
        G, h = s.pair_matrices()
        return {"energies": E, "G": G, "h": h}
    if call == "variance":
        E, var = s.variance()
        return {"moments": np.array([E, var])}
    if call == "renyi":
        return {"entropies": s.correlator(sgs.SGS_CORR_RENYI2, _blocks(case))}
    kind, sites = _sites(case)
    return {"correlator": s.correlator(kind, sites)}


def _sites(case):
    if case["model"] == "kondo":
        return sgs.SGS_CORR_TWO_CHANNEL_K, list(range(1, case["length"]))
    return sgs.SGS_CORR_SPIN_SPIN, list(range(1 + case["bath"]))


# ------------------------------------------------------------------ the same in plain 64-bit torch and numpy

def _quartic(monomials):
    """Antisymmetrised entries ((k, l, p, q), value) of the monomials."""
    out = {}
    for idx, v in monomials:
        for perm in itertools.permutations(range(4)):
            sign = (-1) ** sum(perm[i] > perm[j] for i in range(4) for j in range(i + 1, 4))
            key = tuple(idx[i] for i in perm)
            out[key] = out.get(key, 0.0) + sign * v / 24.0
    return [(k, v) for k, v in out.items() if v != 0.0]


SPIN = np.zeros((3, 4, 4))          # S^a = (i/8) sum K^a_pq c_p c_q on a site's four Majoranas
SPIN[0, 0, 3] = SPIN[2, 0, 1] = 1.0
SPIN[0, 1, 2] = SPIN[1, 0, 2] = SPIN[1, 1, 3] = SPIN[2, 2, 3] = -1.0
SPIN -= SPIN.transpose(0, 2, 1)


def _hamiltonian(case, bath):
    """(A, monomials, constant): H = const + i sum A_kl c_k c_l + sum v c_k c_l c_p c_q."""
    n = _n(case, bath)
    h = np.zeros((n // 2, n // 2))
    const, mono = 0.0, []
    for s in range(2):
        def hop(i, j, x):
            h[2 * i + s, 2 * j + s] = h[2 * j + s, 2 * i + s] = x
        if case["model"] == "kondo":
            L, last = case["length"], 2 * case["length"] - 1
            for ch in range(2):
                for r in range(2, L):
                    hop(1 + 2 * (r - 2) + ch, 1 + 2 * (r - 1) + ch, -case["t"])
                hop(1 + 2 * (L - 2) + ch, last, -case["t"])
        else:
            c = case["channels"]
            hop(0, 0, -case["U"] / 2)
            for ch in range(c):
                hop(0, 1 + ch, -case["V"])
                for r in range(2, bath + 1):
                    hop(1 + (r - 2) * c + ch, 1 + (r - 1) * c + ch, -1.0)
    A = np.zeros((n, n))
    A[0::2, 1::2] = h / 4.0
    A[1::2, 0::2] = -h.T / 4.0
    const += 0.5 * np.trace(h)
    if case["model"] == "kondo":
        for ch in range(2):
            o = 4 * (1 + ch)
            for a in range(3):
                for p, q in itertools.combinations(range(4), 2):
                    for u, v in itertools.combinations(range(4), 2):
                        x = -case["J"] * 4.0 * SPIN[a, p, q] * SPIN[a, u, v] / 64.0
                        if x:
                            mono.append(((p, q, o + u, o + v), x))
    else:
        U = case["U"]
        const += U / 4.0
        for m in range(2):
            A[2 * m, 2 * m + 1] += U / 8.0
            A[2 * m + 1, 2 * m] -= U / 8.0
        mono.append(((0, 1, 2, 3), -U / 4.0))
    return A, mono, const


def _pfaffians(Y):
    """(phase, log|Pf|) of a batch of antisymmetric matrices [B, n, n], by elimination with pivoting."""
    Y = Y.clone()
    B, n, _ = Y.shape
    at = torch.arange(B, device=Y.device)
    phase = torch.ones(B, dtype=torch.complex128, device=Y.device)
    logabs = torch.zeros(B, dtype=torch.float64, device=Y.device)
    for k in range(0, n - 1, 2):
        Z = Y[:, k:, k:]
        p = 1 + Z[:, 1:, 0].abs().argmax(1)
        x, y = Z[at, p].clone(), Z[:, 1].clone()
        Z[at, p] = y
        Z[:, 1] = x
        x, y = Z[at, :, p].clone(), Z[:, :, 1].clone()
        Z[at, :, p] = y
        Z[:, :, 1] = x
        phase = torch.where(p != 1, -phase, phase)
        piv = Z[:, 0, 1].clone()
        phase = phase * piv / piv.abs()
        logabs = logabs + piv.abs().log()
        if k + 2 < n:
            tau, u = Z[:, 0, 2:] / piv[:, None], Z[:, 2:, 1].clone()
            w = tau[:, :, None] * u[:, None, :]
            Z[:, 2:, 2:] += w
            Z[:, 2:, 2:] -= w.transpose(1, 2)
    return phase, logabs


class _Exact:
    """The states of one problem and what follows from them (Sec. II, III of the paper)."""

    def __init__(self, case, bath, gammas):
        self.case, self.g = case, gammas
        A, self.mono, self.const = _hamiltonian(case, bath)
        self.A = torch.from_numpy(A).to(gammas.device)
        self.quartic = _quartic(self.mono)
        M, n = gammas.shape[0], gammas.shape[1]
        self.M, self.n = M, n
        self.pairs = list(itertools.combinations(range(M), 2))
        a = [p for p, _ in self.pairs]
        b = [q for _, q in self.pairs]
        self.index = {pq: i for i, pq in enumerate(self.pairs)}
        Si = torch.linalg.inv(gammas[a] + gammas[b])
        logdet = torch.linalg.slogdet(gammas[a] + gammas[b])[1]
        self.delta = torch.complex(-2.0 * Si, (gammas[a] - gammas[b]) @ Si)          # Delta^{a,b}, a < b
        del Si
        later = [i for i, (p, _) in enumerate(self.pairs) if p > 0]
        phase = torch.ones(len(self.pairs), dtype=torch.complex128, device=gammas.device)
        if later:
            for lo in range(0, len(later), 256):
                part = later[lo:lo + 256]
                phase[part] = case["parity"] * _pfaffians(gammas[0] + self.delta[part])[0]
        mag = torch.exp(0.5 * (-(n // 2) * math.log(2.0) + 0.5 * logdet))
        self.G = np.eye(M, dtype=np.complex128)
        self.h = np.zeros((M, M), dtype=np.complex128)
        gp = (mag * phase).cpu().numpy()
        w = self.wick(self.delta).cpu().numpy()
        wd = self.wick(gammas).cpu().numpy()
        for i, (p, q) in enumerate(self.pairs):
            self.G[p, q], self.G[q, p] = gp[i], gp[i].conj()
            self.h[q, p] = gp[i].conj() * w[i]
            self.h[p, q] = self.h[q, p].conj()
        self.h[np.arange(M), np.arange(M)] = wd
        self.solve()

    def wick(self, D):
        e = self.const + (self.A.T * D).sum((1, 2))
        for (k, l, p, r), v in self.quartic:
            e = e - 3.0 * v * D[:, k, l] * D[:, p, r]
        return e

    def solve(self):
        w, U = np.linalg.eigh(self.G)
        keep = w > 1e-12 * w.max()
        X = U[:, keep] / np.sqrt(w[keep])
        H = X.conj().T @ self.h @ X
        e, V = np.linalg.eigh(0.5 * (H + H.conj().T))
        lam = X @ V[:, 0]
        lam = lam / math.sqrt((lam.conj() @ self.G @ lam).real)
        j = int(np.argmax(np.abs(lam)))
        self.E, self.lam = float(e[0]), lam * (abs(lam[j]) / lam[j])

    def transition(self, b, a):
        """Delta^{b,a}: <phi_a| . |phi_b>."""
        if a == b:
            return self.g[a].to(torch.complex128)
        return self.delta[self.index[b, a]] if b < a else self.delta[self.index[a, b]].conj()

    def derivative(self, mu):
        lt = self.G @ self.lam
        z = self.lam[mu] * lt[mu].conjugate()
        c = z.conjugate() / abs(z) if self.case["phase_c"] else 1.0 / z
        acc = torch.zeros(self.n, self.n, dtype=torch.complex128, device=self.g.device)
        for be in range(self.M):
            D = self.transition(be, mu)
            F = self.A.to(torch.complex128)
            for (k, l, m, r), v in self.quartic:
                F[k, l] += 6.0 * v * D[m, r]
            DF = D @ F
            G, lam = complex(self.G[mu, be]), complex(self.lam[be])
            acc += lam * (2j * G * (DF - DF.T) + 2.0 * G * (DF @ D + F) - (complex(self.h[mu, be]) - self.E * G) * D)
        return 2.0 * (complex(lt[mu].conjugate() * c) * acc).real

    def stepped(self):
        out = []
        for mu in range(self.M):
            g, d = self.g[mu], self.derivative(mu)
            X = g @ d
            R = torch.linalg.matrix_exp(0.25 * self.case["dtau"] * (X - X.T))       # d g = (g d)^T
            x = R @ g @ R.T
            x = 0.5 * (x - x.T)
            for _ in range(2):
                x = 1.5 * x + 0.5 * x @ (x @ x)
                x = 0.5 * (x - x.T)
            out.append(x)
        return torch.stack(out)

    def terms(self):
        """(conj(lambda_a) lambda_b G_ab, Delta^{b,a}) of every ordered pair."""
        for a in range(self.M):
            for b in range(self.M):
                yield complex(self.lam[a].conjugate() * self.lam[b] * self.G[a, b]), self.transition(b, a)

    def spin(self, sites):
        tot = np.zeros(len(sites), dtype=np.complex128)
        for w, D in self.terms():
            D = D.resolve_conj().cpu().numpy()
            B00 = D[:4, :4]
            for i, s in enumerate(sites):
                if s == 0:
                    pf = B00[0, 1] * B00[2, 3] - B00[0, 2] * B00[1, 3] + B00[0, 3] * B00[1, 2]
                    tot[i] += w * 3.0 / 8.0 * (1.0 - pf)
                    continue
                B0s, Bss = D[:4, 4 * s:4 * s + 4], D[4 * s:4 * s + 4, 4 * s:4 * s + 4]
                for K in SPIN:
                    x = (K * B00).sum() * (K * Bss).sum() - 2.0 * np.einsum("pq,uv,pu,qv", K, K, B0s, B0s)
                    tot[i] += w * x / 64.0
        return tot.real

    def variance(self):
        tot = 0.0
        eye = torch.eye(self.n, dtype=torch.complex128, device=self.g.device)
        A = self.A.to(torch.complex128)
        (idx, v), e = self.mono[0], self.const          # one quartic term

        def pf(X):
            s, l = _pfaffians(X[None])
            return complex(s[0]) * math.exp(float(l[0]))

        def ordered(g, ix):
            X = torch.triu(g[ix][:, ix], 1)
            return X - X.T
        for w, D in self.terms():
            g = eye + 1j * D
            AD = A @ D
            T = complex(AD.diagonal().sum())
            h2 = e * e + T * T - 2.0 * complex((A * A.T).sum()) - 2.0 * complex((AD * AD.T).sum())
            B, Bp = g.T @ A @ g, g @ A @ g.T
            x, ix = ordered(g, list(idx)), list(idx)
            p4 = complex(x[0, 1] * x[2, 3] - x[0, 2] * x[1, 3] + x[0, 3] * x[1, 2])
            h2 += 2.0 * e * (T + v * p4)
            for C in (B - B.T, Bp - Bp.T):
                c = C[ix][:, ix]
                d = complex(c[0, 1] * x[2, 3] + x[0, 1] * c[2, 3] - c[0, 2] * x[1, 3] - x[0, 2] * c[1, 3]
                            + c[0, 3] * x[1, 2] + x[0, 3] * c[1, 2])
                h2 += v * (T * p4 - 1j * d)
            h2 += v * v * pf(ordered(g, ix + ix))
            tot += (w * h2).real
        return tot - self.E ** 2

    def renyi(self, l):
        m = 4 * (1 + l)
        pairs = list(itertools.product(range(self.M), repeat=2))
        B = torch.stack([self.transition(a, b)[:m, :m] for a, b in pairs])
        w = torch.tensor([complex(self.lam[a] * self.lam[b].conjugate() * self.G[b, a]) for a, b in pairs],
                         dtype=torch.complex128, device=B.device)
        one = 1j * torch.eye(m, dtype=torch.complex128, device=B.device)
        tot = 0.0
        for u in range(len(pairs)):
            Z = torch.zeros(len(pairs), 2 * m, 2 * m, dtype=torch.complex128, device=B.device)
            Z[:, :m, :m] = B[u]
            Z[:, m:, m:] = B
            Z[:, :m, m:] = one
            Z[:, m:, :m] = -one
            ph, la = _pfaffians(Z)
            tot += float((w[u] * w * ph * torch.exp(la - (m // 2) * math.log(2.0))).sum().real)
        return -math.log(tot)


def exact(case, seed):
    if case["call"] == "step" and _n(case, case["bath"]) > 1000 and case["rank"] > 8:
        return None
    got, energies = {}, []
    for i, (bath, M) in enumerate(_problems(case)):
        g = _states(_n(case, bath), M, seed * 64 + i, case["parity"])
        x = _Exact(case, bath, g)
        if case["call"] in ("step", "serve"):
            E = [x.E]
            for _ in range(case["steps"] - 1):
                x = _Exact(case, bath, x.stepped())
                E.append(x.E)
            energies.append(E)
            got[f"gamma{i}"], got[f"lambda{i}"] = x.stepped(), x.lam
    if case["call"] in ("step", "serve"):
        return {"energies": np.array(energies), **got}
    if case["call"] == "energy":
        return {"energies": np.array([x.E]), "G": x.G, "h": x.h}
    if case["call"] == "variance":
        return {"moments": np.array([x.E, x.variance()])}
    if case["call"] == "renyi":
        return {"entropies": np.array([x.renyi(l) for l in _blocks(case)])}
    sites = _sites(case)[1]
    if case["model"] == "kondo":
        return {"correlator": x.spin([2 * r - 1 for r in sites]) + x.spin([2 * r for r in sites])}
    return {"correlator": x.spin(sites)}
