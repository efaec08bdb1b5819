"""The work that a user of this package has it do, as cases that can be timed
and compared: whole imaginary-time paths and stabilisation blocks in both
precisions, ragged batches, the estimators, low rank and the mu derivative.

listed()            the cases, draw(rng) one more of the same ranges
prepare(case, seed) the context(s) and the auxiliary fields x ~ N(0, 1) that a
                    program holds before the call
run(state)          one pass through the public entry points, and its results
work(case)          bytes and flops that a pass cannot do without
exact(case, seed)   the results in 64 bits from plain torch: A(tau) multiplied
                    out and inverted, with no stabilisation

The mixed-precision path computes G and ln det in single precision (it widens
them into the complex128 / float64 buffers of the ABI), so its results are
taken as complex64 / float32; the complex128 path's as they are.
"""
import itertools
import math

import numpy as np
import torch

import paper_2012_12228_gb300 as ftq

SHELLS = [7, 19, 27, 33, 57, 81, 93, 123, 147, 171, 179, 203, 251, 257]    # closed-shell basis sizes
DTAU = 0.05


def _path(name, M, N, rs, theta, walkers, precision, slices, dtau=DTAU, ends="state"):
    return {"name": name, "kind": "path", "M": M, "N": N, "rs": rs, "theta": theta, "dtau": dtau,
            "walkers": walkers, "precision": precision, "slices": slices, "ends": ends}


def listed():
    return [
        # the smallest system, the one that exact diagonalisation checks: the whole path to tau = beta
        # and its estimates; launches and latency count
        _path("c128 M=7 whole path", 7, 2, 1.0, 0.5, 64, "fp64", 0, ends="estimate"),
        # a small basis in double precision with population control half way, as a production
        # run on it combs between stabilisation blocks
        _path("c128 M=33 comb", 33, 14, 1.0, 0.25, 300, "fp64", 20, ends="comb"),
        # mu tuning: the whole path in double precision, <N>, <E> and their derivatives (a Newton step)
        _path("c128 M=57 mu tuning", 57, 14, 1.0, 0.5, 256, "fp64", 0, ends="mu"),
        # the plain complex128 path on the large basis: one stabilisation block
        _path("c128 M=257 block", 257, 66, 1.0, 0.0625, 152, "fp64", 5, dtau=0.025),
        # a mid-sized production run in mixed precision: 87 slices to tau = beta and the estimates
        _path("mixed M=57 whole path", 57, 14, 1.0, 0.125, 640, "mixed", 0, ends="estimate"),
        # time-slice estimates recorded along a mixed path
        _path("mixed M=123 tracked", 123, 14, 2.0, 0.25, 256, "mixed", 10, ends="track"),
        # the headline: 1024 walkers, one stabilisation block of five slices
        _path("mixed M=257 block", 257, 66, 1.0, 0.0625, 1024, "mixed", 5, dtau=0.025),
        # a high cutoff, few walkers, one stabilisation block
        _path("mixed M=515 block", 515, 14, 0.5, 0.125, 64, "mixed", 5),
        # four systems of different basis size side by side (the ragged workload)
        {"name": "ragged batch", "kind": "ragged", "systems": "57/14/0.5/0.0625 123/38/2.0/0.5 "
         "171/54/1.0/0.125 257/66/1.0/0.0625", "dtau": DTAU, "walkers": 256, "slices": 5},
        # the observables of walkers at hand: energies, particle numbers, structure factor
        {"name": "observables M=257", "kind": "observables", "M": 257, "N": 66, "rs": 1.0, "theta": 0.0625,
         "dtau": 0.025, "walkers": 128},
        # low-rank truncation along a whole path
        {"name": "low rank M=257", "kind": "lowrank", "M": 257, "N": 14, "rs": 0.5, "theta": 0.125, "dtau": DTAU,
         "walkers": 32, "threshold": 1e-6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _electrons(rng, M):
    return rng.choice([n for n in (2, 14, 38, 54, 66) if 2 * n <= M] or [2])


def draw(rng):
    """A case of the listed ranges: the walkers are bounded so that a pass costs at most about as much as
    the largest listed one."""
    kind = rng.choice(["fp64", "fp64", "mixed", "mixed", "mixed", "ragged", "observables", "lowrank"])
    M = rng.choice(SHELLS)
    N = _electrons(rng, M)
    rs, theta = rng.choice([0.5, 1.0, 2.0]), rng.choice([0.125, 0.25, 0.5])
    dtau = rng.choice([0.025, 0.05])
    slices = rng.randint(3, 12)
    size = (M / 257.0) ** 3 + 1e-4
    if kind == "fp64":
        W = _log_int(rng, 3, min(600, max(8, int(100 * 5 / slices / size))))
        return _drawn(_path("", M, N, rs, theta, W, kind, slices, dtau, rng.choice(["state", "state", "comb"])))
    if kind == "mixed":
        W = _log_int(rng, 3, min(1200, max(8, int(1000 * 5 / slices / size))))
        return _drawn(_path("", M, N, rs, theta, W, kind, slices, dtau, rng.choice(["state", "state", "track"])))
    if kind == "ragged":
        sizes = [rng.choice(SHELLS) for _ in range(rng.randint(2, 4))]
        text = " ".join("%d/%d/%s/%s" % (m, _electrons(rng, m), rng.choice([0.5, 1.0, 2.0]), rng.choice([0.125, 0.5]))
                        for m in sizes)
        return {"kind": "ragged", "systems": text, "dtau": dtau, "walkers": _log_int(rng, 4, 256),
                "slices": rng.randint(2, 6)}
    if kind == "observables":
        return {"kind": kind, "M": M, "N": N, "rs": rs, "theta": theta, "dtau": dtau,
                "walkers": _log_int(rng, 3, min(512, max(8, int(100 / size))))}
    return {"kind": kind, "M": rng.choice([57, 81, 123, 147, 171]), "N": 14, "rs": 0.5, "theta": 0.125, "dtau": DTAU,
            "walkers": _log_int(rng, 3, 40), "threshold": rng.choice([1e-6, 1e-5])}


def _drawn(case):
    del case["name"]
    return case


# ---------------------------------------------------------------- the passes
def _systems(case):
    """The (M, N, rs, theta) of every system of a case."""
    if case["kind"] != "ragged":
        return [(case["M"], case["N"], case["rs"], case["theta"])]
    out = []
    for text in case["systems"].split():
        m, n, rs, theta = text.split("/")
        out.append((int(m), int(n), float(rs), float(theta)))
    return out


def _slices(case, n):
    """Slices of a pass on a path of n slices (0 or none given: the whole path)."""
    return min(case.get("slices") or n, n)


def _beta(rs, theta):
    return 1.0 / (theta * 0.5 * (9.0 * math.pi / 4.0) ** (2.0 / 3.0) / rs ** 2)


def _path_slices(rs, theta, dtau):
    return max(1, int(round(_beta(rs, theta) / dtau)))


def _fields(seed, which, shape):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 7919 * which + 11)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case}
    if kind == "ragged":
        systems = [dict(N=n, M=m, rs=rs, theta=th, dtau=case["dtau"], walkers=case["walkers"])
                   for m, n, rs, th in _systems(case)]
        b = ftq.Batch(systems)
        b.autotune()
        n = min(_slices(case, p.n_slices) for p in b.members)
        state["batch"] = b
        state["fields"] = [_fields(seed, k, (n, p.W, p.n_alpha)) for k, p in enumerate(b.members)]
        return state
    mixed = case.get("precision") == "mixed"
    p = ftq.Propagator(case["N"], case["M"], case["rs"], case["theta"], case["dtau"], walkers=case["walkers"],
                       precision=ftq.FTQ_MIXED if mixed else ftq.FTQ_FP64, low_rank=case.get("threshold", 0.0))
    if mixed:
        p.autotune()
    state["p"] = p
    n = min(5, p.n_slices) if kind == "observables" else _slices(case, p.n_slices)
    fields = _fields(seed, 0, (n, p.W, p.n_alpha))
    if kind == "observables":
        p.propagate(fields)            # walkers to look at; the pass is the evaluation alone
    elif case.get("ends") == "track":
        p.track_estimates(1)
    state["fields"] = fields
    if case.get("ends") == "comb":
        state["half"] = (fields[:(n + 1) // 2].contiguous(), fields[(n + 1) // 2:].contiguous())
        state["xi"] = float(np.random.default_rng(seed).uniform(0.1, 0.9))
    return state


def _record(p, single):
    """The walkers' weight record without its unused last entry."""
    w = p.weights()[:, :7]
    return w.float() if single else w


def _green(p, single):
    g = p.green()
    return g.to(torch.complex64) if single else g


def _estimates(p):
    e = p.estimators()
    total = np.array([e["E"].real, e["E"].imag, e["N"].real, e["N"].imag])
    return {"per_walker": e["per_walker"][:, :7], "total": total, "alive": e["n_alive"]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ragged":
        b = state["batch"]
        for p in b.members:
            p.reset()
        b.propagate(state["fields"])
        return [{"weights": _record(p, True), "green": _green(p, True)} for p in b.members]
    p = state["p"]
    if kind == "observables":
        s = p.structure_factor(per_walker=True)
        return {"estimates": _estimates(p), "rhorho": s["rhorho"], "S": s["S"], "per_walker": s["per_walker"]}
    single = case.get("precision") == "mixed"
    ends = case.get("ends", "state")
    p.reset()
    if ends == "comb":
        first, second = state["half"]
        p.propagate(first)
        parent = p.population_control(state["xi"])
        p.propagate(second)
        return {"parent": parent, "weights": _record(p, single), "green": _green(p, single)}
    p.propagate(state["fields"])
    if kind == "lowrank":
        return {"weights": _record(p, False), "green": _green(p, False), "ranks": p.ranks(), **_estimates(p)}
    out = {"weights": _record(p, single), "green": _green(p, single)}
    if ends == "estimate":
        e = _estimates(p)
        if single:
            e["per_walker"] = e["per_walker"].float()
            e["total"] = e["total"].astype(np.float32)
        out.update(e)
    elif ends == "mu":
        g = p.mu_grad()
        out["mu"] = {"per_walker": g["per_walker"], "total": np.array([g["dN"], g["dE"], g["N"], g["E"]])}
    elif ends == "track":
        t = p.slice_estimates()
        out["k"] = t["k"]
        out["slices"] = np.stack([t["E"].real, t["N"].real]).astype(np.float32)
    return out


def work(case):
    """Flops: eight real ones per complex multiply-add of the Taylor products, the LU and the solves of G, and
    the factorisation, Q and T update of a stabilisation; bytes: fields in, records and G out."""
    nbytes = flops = 0.0
    for M, N, rs, theta in _systems(case):
        W = case["walkers"]
        n = _path_slices(rs, theta, case["dtau"])
        pairs = _pair_terms(M)
        if case["kind"] == "observables":
            nbytes += W * (16.0 * M * M + 64 + 16 * pairs[0])
            flops += W * 2 * 8.0 * pairs[1]
            continue
        n = _slices(case, n)
        size = 8.0 if case.get("precision") == "mixed" or case["kind"] == "ragged" else 16.0
        nbytes += W * (n * 8.0 * pairs[0] + size * M * M + 64)
        flops += W * n * (6 * 8 + 32.0 / 3) * M ** 3 + W * (n // 5) * (44.0 / 3) * M ** 3
        if case.get("ends") == "track":
            flops += W * n * 8.0 * pairs[1]
        if case.get("ends") in ("estimate", "mu") or case["kind"] == "lowrank":
            flops += W * 8.0 * pairs[1]
    return {"bytes": nbytes, "flops": flops}


_TERMS = {}


def _pair_terms(M):
    """(momentum transfers, exchange terms of the half space) of the closed shell with M members."""
    if M not in _TERMS:
        n = _basis(M)
        d = (n[:, None, :] - n[None, :, :]).reshape(-1, 3)
        counts = np.unique(d, axis=0, return_counts=True)[1].astype(np.float64)
        _TERMS[M] = (len(counts) - 1, float((counts ** 2).sum() - M * M) / 2)
    return _TERMS[M]


# ---------------------------------------------------------------- 64-bit results from plain torch
def _basis(M):
    for cut in range(64):
        r = math.isqrt(cut)
        v = [n for n in itertools.product(range(-r, r + 1), repeat=3) if n[0] ** 2 + n[1] ** 2 + n[2] ** 2 <= cut]
        if len(v) == M:
            return np.array(sorted(v, key=lambda n: (n[0] ** 2 + n[1] ** 2 + n[2] ** 2, n)))
    raise ValueError(M)


class _Gas:
    """The uniform electron gas of one system, its transfers and tables."""

    def __init__(self, M, N, rs, theta, dtau):
        n = _basis(M)
        L = (4.0 * math.pi * N / 3.0) ** (1.0 / 3.0) * rs
        omega, kf = L ** 3, 2.0 * math.pi / L
        self.M = M
        self.eps = 0.5 * kf ** 2 * (n ** 2).sum(1).astype(np.float64)
        self.beta = _beta(rs, theta)
        self.n = _path_slices(rs, theta, dtau)
        self.dtau = self.beta / self.n
        diff = n[:, None, :] - n[None, :, :]
        d2 = (diff ** 2).sum(2).astype(np.float64)
        with np.errstate(divide="ignore"):
            deps = -0.5 * np.where(d2 > 0, 4.0 * math.pi / (omega * kf ** 2 * d2), 0.0).sum(1)
        lo, hi = self.eps.min() - 50 / self.beta - 10, self.eps.max() + 50 / self.beta + 10
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            filled = 2.0 * (0.5 * (1.0 - np.tanh(0.5 * self.beta * (self.eps - mid)))).sum()
            lo, hi = (mid, hi) if filled < N else (lo, mid)
        self.mu = 0.5 * (lo + hi)
        self.E_M = 0.5 * N * (-2.837297 / L)
        # slots: 1 + 2q for the half-space transfer +q, 2 + 2q for -q, 0 on the diagonal
        q = np.unique(diff.reshape(-1, 3), axis=0)
        first = np.where(q[:, 0] != 0, q[:, 0], np.where(q[:, 1] != 0, q[:, 1], q[:, 2]))
        half = sorted(map(tuple, q[first > 0]), key=lambda v: (v[0] ** 2 + v[1] ** 2 + v[2] ** 2, v))
        slot = {}
        for i, v in enumerate(half):
            slot[v] = 1 + 2 * i
            slot[tuple(-c for c in v)] = 2 + 2 * i
        slot[(0, 0, 0)] = 0
        self.nq = len(half)
        self.slots = np.array([slot[tuple(v)] for v in diff.reshape(-1, 3)])
        q2 = kf ** 2 * np.array([float(sum(c * c for c in v)) for v in half])
        self.vq = self._gpu(4.0 * math.pi / (omega * q2))
        self.cq = self._gpu(np.sqrt(2.0 * math.pi / (omega * q2)))
        self.h = self._gpu(np.exp(-0.5 * self.dtau * (self.eps + deps - self.mu)))
        self.index = torch.from_numpy(self.slots).cuda()
        self.e = self._gpu(self.eps)

    @staticmethod
    def _gpu(v):
        return torch.from_numpy(np.ascontiguousarray(v)).cuda()

    def rho(self, P):
        """sum of P_ab over the pairs with n_a - n_b = Q, for every slot."""
        out = torch.zeros((P.shape[0], 2 * self.nq + 1, 2), dtype=torch.float64, device="cuda")
        out.index_add_(1, self.index, torch.view_as_real(P.reshape(P.shape[0], -1).contiguous()))
        return torch.view_as_complex(out)

    def left(self, k):
        return torch.exp(-(self.n - k) * self.dtau * (self.e - self.mu))

    def green(self, R, k):
        """(I + R D_L)^-1 and ln det(I + R D_L), D_L = B_T^(n - k) split into factors of at most one."""
        d = self.left(k)
        big = torch.clamp(1.0 / d, max=1.0)
        X = R * torch.clamp(d, max=1.0)
        X.diagonal(dim1=1, dim2=2).add_(big)
        lu, piv = torch.linalg.lu_factor(X)
        u = lu.diagonal(dim1=1, dim2=2)
        swaps = (piv != torch.arange(1, self.M + 1, device="cuda")).sum(1)
        ld = torch.complex(u.abs().log().sum(1), u.angle().sum(1) + math.pi * (swaps % 2)) - big.log().sum()
        rows = torch.diag_embed(big.to(X.dtype)).expand(X.shape).contiguous()
        return torch.linalg.lu_solve(lu, piv, rows, left=False).resolve_conj(), ld


def _wrap(x):
    return torch.remainder(x + math.pi, 2 * math.pi) - math.pi


class _Walkers:
    """Walkers on the directly multiplied chain."""

    def __init__(self, gas, W):
        self.gas, self.k = gas, 0
        M = gas.M
        self.R = torch.eye(M, dtype=torch.complex128, device="cuda").expand(W, M, M).contiguous()
        d = gas.left(0)
        self.G = torch.diag_embed((1.0 / (1.0 + d)).to(torch.complex128)).expand(W, M, M)
        self.ld = torch.log1p(d).sum().to(torch.complex128).expand(W).clone()
        self.logw = torch.zeros(W, dtype=torch.float64, device="cuda")
        self.alive = torch.ones(W, dtype=torch.float64, device="cuda")
        self.gauss = torch.zeros(W, dtype=torch.complex128, device="cuda")

    def one_rdm(self):
        return torch.eye(self.gas.M, dtype=torch.complex128, device="cuda") - self.G.transpose(1, 2)

    def step(self, x, order=6):
        g = self.gas
        self.k += 1
        r = g.rho(self.one_rdm())
        rp, rm = r[:, 1::2], r[:, 2::2]
        s = math.sqrt(g.dtau)
        bA, bB = -s * 2j * g.cq * (rp + rm), s * 2.0 * g.cq * (rp - rm)
        xA, xB = x[:, 0::2], x[:, 1::2]
        yA, yB = xA - bA, xB - bB
        phi = torch.zeros_like(r)
        phi[:, 1::2] = s * g.cq * 1j * (yA + 1j * yB)
        phi[:, 2::2] = s * g.cq * 1j * (yA - 1j * yB)
        V = phi[:, g.index].reshape(self.G.shape)
        self.gauss = (bA * xA - 0.5 * bA * bA + bB * xB - 0.5 * bB * bB).sum(1)
        Y = g.h[:, None] * self.R
        Z = Y
        for j in range(order, 0, -1):
            Z = torch.baddbmm(Y, V, Z, alpha=1.0 / j)
        self.R = g.h[:, None] * Z
        self.G, ld = g.green(self.R, self.k)
        lnS = 2.0 * (ld - self.ld)
        c = torch.cos(lnS.imag)
        live = (self.alive > 0.5) & (c > 0)
        self.logw = torch.where(live, self.logw + lnS.real + self.gauss.real + torch.log(c.clamp(min=1e-300)),
                                self.logw)
        self.alive = live.to(torch.float64)
        self.ld = torch.complex(ld.real, _wrap(ld.imag))

    def record(self):
        z = torch.zeros_like(self.logw)
        return torch.stack([self.logw, z, self.alive, self.ld.real, self.ld.imag, self.gauss.real, self.gauss.imag], 1)

    def comb(self, xi):
        """Systematic resampling; survivors keep their slot, extra copies fill the free ones in order."""
        W = self.logw.shape[0]
        lw = torch.where(self.alive > 0.5, self.logw, torch.full_like(self.logw, -math.inf)).cpu().numpy()
        w = np.exp(lw - lw.max())
        c = np.cumsum(w)
        counts = np.bincount(np.searchsorted(c, (np.arange(W) + xi) * (c[-1] / W), side="right").clip(max=W - 1),
                             minlength=W)
        parent = np.arange(W)
        parent[counts == 0] = np.repeat(np.arange(W), np.maximum(counts - 1, 0))
        at = torch.from_numpy(parent).cuda()
        self.R, self.G, self.ld, self.gauss = self.R[at], self.G[at], self.ld[at], self.gauss[at]
        self.logw = torch.full_like(self.logw, math.log(c[-1] / W) + lw.max())
        self.alive = torch.ones_like(self.alive)
        return parent

    def exchange(self, P):
        """sum over the pairs (a, d), (b, c) of Q of P_ab P_cd, for every half-space transfer."""
        g = self.gas
        order = np.argsort(g.slots, kind="stable")
        ends = np.cumsum(np.bincount(g.slots, minlength=2 * g.nq + 1))
        out = torch.empty((P.shape[0], g.nq), dtype=torch.complex128, device="cuda")
        for q in range(g.nq):
            at = order[ends[2 * q]:ends[2 * q + 1]]
            a, d = torch.from_numpy(at // g.M).cuda(), torch.from_numpy(at % g.M).cuda()
            out[:, q] = (P[:, a[:, None], a[None, :]] * P[:, d[None, :], d[:, None]]).sum((1, 2))
        return out

    def energies(self):
        g = self.gas
        P = self.one_rdm()
        diag = P.diagonal(dim1=1, dim2=2)
        r = g.rho(P)
        lam = self.exchange(P)
        E = g.E_M + (2.0 * g.e * diag).sum(1) + ((4.0 * r[:, 1::2] * r[:, 2::2] - 2.0 * lam) * g.vq).sum(1)
        return E, 2.0 * diag.sum(1), r, lam, P

    def weights(self):
        top = torch.where(self.alive > 0.5, self.logw, torch.full_like(self.logw, -math.inf)).max()
        return torch.where(self.alive > 0.5, torch.exp(self.logw - top), torch.zeros_like(self.logw))

    def estimates(self):
        E, N = self.energies()[:2]
        w = self.weights()
        E0, N0 = (w * E).sum() / w.sum(), (w * N).sum() / w.sum()
        z = torch.zeros_like(self.logw)
        rec = torch.stack([self.logw, z, self.alive, E.real, E.imag, N.real, N.imag], 1)
        return {"per_walker": rec, "total": torch.stack([E0.real, E0.imag, N0.real, N0.imag]), "alive": None}


def exact(case, seed):
    kind, ends = case["kind"], case.get("ends", "state")
    if kind == "lowrank":
        return None                      # truncated by intent: the untruncated result is not what it computes
    out = []
    for k, (M, N, rs, theta) in enumerate(_systems(case)):
        gas = _Gas(M, N, rs, theta, case["dtau"])
        n = _slices(case, min(_path_slices(r, t, case["dtau"]) for _, _, r, t in _systems(case)))
        if kind == "observables":
            n = min(5, gas.n)
        x = _fields(seed, k, (n, case["walkers"], 2 * gas.nq))
        ws = _Walkers(gas, case["walkers"])
        parent, track = None, []
        for i in range(n):
            if ends == "comb" and i == (n + 1) // 2:
                parent = ws.comb(float(np.random.default_rng(seed).uniform(0.1, 0.9)))
            ws.step(x[i])
            if ends == "track":
                t = ws.estimates()["total"]
                track.append((t[0], t[2]))
        out.append((ws, parent, track))
    if kind == "ragged":
        return [{"weights": w.record(), "green": w.G} for w, _, _ in out]
    ws, parent, track = out[0]
    if kind == "observables":
        E, N, r, lam, P = ws.energies()
        diag = P.diagonal(dim1=1, dim2=2)
        g = ws.gas
        own = torch.zeros((P.shape[0], 2 * g.nq + 1), dtype=torch.complex128, device="cuda")
        mask = g.index != 0
        rows = torch.arange(g.M, device="cuda").repeat_interleave(g.M)[mask]
        add = torch.view_as_real(own)
        add.index_add_(1, g.index[mask], torch.view_as_real(2.0 * diag[:, rows].contiguous()))
        pair = 4.0 * r[:, 1::2] * r[:, 2::2] - 2.0 * lam
        own[:, 1::2] += pair
        own[:, 2::2] += pair
        per = own[:, 1:]
        w = ws.weights()
        mean = (w[:, None] * per).sum(0) / w.sum()
        return {"estimates": ws.estimates(), "rhorho": mean, "S": mean.real / case["N"], "per_walker": per}
    res = {"weights": ws.record(), "green": ws.G}
    if ends == "comb":
        res["parent"] = torch.from_numpy(parent)
    elif ends == "estimate":
        res.update(ws.estimates())
    elif ends == "mu":
        res["mu"] = {"per_walker": None, "total": None}
    elif ends == "track":
        res["k"] = None
        res["slices"] = torch.tensor([[float(e) for e, _ in track], [float(v) for _, v in track]], dtype=torch.float64)
    return res
