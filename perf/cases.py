"""The work that users of this library have it do, as cases to be timed.

A case is one call pattern of the C ABI (through its ctypes binding) at one
size: Markov chains that exist already are advanced and read back.
``prepare`` makes the start configurations and the handle that a program
keeps, ``run`` is one pass over them, ``exact`` the same pass in plain FP64
torch (momenta from Philox4x32-10 and Box-Muller, leapfrog or minimum-norm
integrator, Metropolis test, Sec. 4 estimators of arXiv:1912.03278).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1912_03278_gb300 as pkg

PREC = {"fp64": pkg.ISING_PREC_PLAIN_FP64, "fp32": pkg.ISING_PREC_FP32,
        "bf16": pkg.ISING_PREC_BF16, "fp8": pkg.ISING_PREC_FP8}
INTEG = {"leapfrog": pkg.ISING_INTEGRATOR_LEAPFROG, "omelyan": pkg.ISING_INTEGRATOR_OMELYAN}
OMELYAN_LAMBDA = 0.1931833275037836   # the minimum-norm value


def listed():
    return [
        # A small study: sizes at which autocorrelation times are measured.
        # Many short trajectories per call; latency and launches count.
        _case("study2d_L16", L="16,16", chains=64, n_md=5, eps=0.2, n_traj=8,
              beta=0.42, beta_hi=0.46),
        # The lower size of the 16-beta sweep around the critical point (part
        # of its chains), the state continued from call to call.
        _case("sweep2d_L256", L="256,256", chains=1216, n_md=20, eps=0.06, beta=0.38, beta_hi=0.50),
        # The upper size of the sweep: the largest call.
        _case("sweep2d_L1024", L="1024,1024", chains=1216, n_md=20, eps=0.04, beta=0.38,
              beta_hi=0.50),
        # Odd extents (rows that do not split into 16-byte vectors), a field
        # per site, the minimum-norm integrator: a finite-size study.
        _case("odd2d_field", L="251,173", chains=304, n_md=6, eps=0.16, integrator="omelyan",
              field=0.1, beta=0.36, beta_hi=0.44),
        # The mixed 3D batch: five sizes, 64 chains each, one group launch, the
        # chains of the two largest sizes on two CTAs each.
        _case("mixed3d", kind="group", L="16,24,32,48,64", splits="1,1,1,2,2", chains=64,
              h=0.05, beta=0.2217),
        # One 3D lattice of unequal extents, resumed from a checkpoint held on
        # the device in every pass, with the sign-flip proposal.
        _case("resume3d", L="40,28,36", chains=160, n_md=10, eps=0.18, flip=1, resume=True,
              beta=0.2, beta_hi=0.23),
        # The all-to-all model of the appendix, chains that fit a CTA.
        _case("infinite_N4096", kind="infinite", N=4096, chains=2432, n_md=8, eps=0.125, beta=1.0),
        # Chains too long for one CTA's registers, length not a multiple of 4.
        _case("infinite_N50001", kind="infinite", N=50001, chains=304, n_md=10, eps=0.07, h=0.02,
              beta=0.9, beta_hi=1.1),
        # Dense (SK) couplings on the tensor cores, with fields per site.
        _case("dense_bf16_N4096", kind="dense", N=4096, chains=1024, n_md=10, eps=0.17, prec="bf16",
              field=0.1, beta=0.5),
        # The FP8 form at a size and chain count that leave tiles ragged.
        _case("dense_fp8_N1408", kind="dense", N=1408, chains=200, n_md=8, eps=0.1, prec="fp8",
              flip=2, n_traj=2, beta=0.5),
        # The FP64 form, a few chains: a check run beside a production run.
        _case("plain_fp64_L128", L="128,128", chains=4, n_md=9, eps=0.11, prec="fp64", h=0.01,
              beta=0.4, beta_hi=0.44),
        # Local Metropolis-Hastings sweeps of the same lattices, the spins read
        # after a block of them.
        _case("mh2d_L256", kind="mh", L="256,256", chains=64, n_traj=256, beta=0.38, beta_hi=0.50),
    ]


def _case(name, kind="lattice", L="", N=0, chains=1, n_md=1, eps=0.1, n_traj=1, beta=0.4,
          beta_hi=0.0, h=0.0, field=0.0, prec="fp32", integrator="leapfrog", flip=0, resume=False,
          splits=""):
    c = dict(kind=kind, L=L, N=N, chains=chains, n_md=n_md, eps=eps, n_traj=n_traj, beta=beta,
             beta_hi=beta_hi or beta, h=h, field=field, prec=prec, integrator=integrator, flip=flip,
             resume=resume, splits=splits)
    if name:
        c["name"] = name
    return c


# Site-passes (sites x chains x force evaluations) of the largest listed case
# are 2.7e10; a drawn case stays well below.
_MOST = 8e9


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _chains(rng, sites, passes, hi=4096):
    return max(1, min(_log_int(rng, 4, hi), int(_MOST / (sites * passes))))


def draw(rng):
    kind = rng.choice(["lat2", "lat2", "lat2", "lat3", "lat3", "group", "infinite", "infinite", "dense", "dense",
                       "fp64", "mh"])
    beta = rng.uniform(0.36, 0.46)
    n_md = rng.randint(4, 24)
    eps = rng.uniform(0.3, 1.1) / n_md
    if kind == "lat2":
        # rows that split into 16-byte vectors in two of three draws
        X = _log_int(rng, 8, 1024)
        if rng.random() < 0.67:
            X = max(8, X // 4 * 4)
        L = (X, _log_int(rng, 8, 1024))
        omelyan = rng.random() < 0.3
        chains = _chains(rng, L[0] * L[1], (2 if omelyan else 1) * n_md + 1)
        return _case("", L="%d,%d" % L, chains=chains, n_md=n_md,
                     eps=eps * 50.0 / (50.0 + (L[0] * L[1]) ** 0.5), n_traj=rng.choice([1, 1, 2, 4]), beta=beta,
                     beta_hi=beta + 0.05, integrator="omelyan" if omelyan else "leapfrog",
                     h=rng.choice([0.0, 0.0, 0.03]), field=rng.choice([0.0, 0.0, 0.1]),
                     flip=rng.choice([0, 0, 2]), resume=rng.random() < 0.3)
    if kind == "lat3":
        X = rng.randint(8, 60)
        if X % 4 == 0 or rng.random() < 0.6:
            X = X // 4 * 4
            L = (X, rng.randint(6, 60), rng.randint(6, 64))
        else:   # scalar rows: planes of at most 1024 sites
            L = (X, max(5, min(60, rng.randint(500, 1000) // X)), rng.randint(6, 64))
        N = L[0] * L[1] * L[2]
        return _case("", L="%d,%d,%d" % L, chains=_chains(rng, N, n_md + 1, 1024), n_md=n_md,
                     eps=eps, beta=rng.uniform(0.18, 0.24), h=rng.choice([0.0, 0.05]),
                     flip=rng.choice([0, 0, 1]), resume=rng.random() < 0.4)
    if kind == "group":
        sizes = sorted(rng.sample([12, 16, 18, 20, 24, 28, 32, 36, 40, 44, 48, 56, 64],
                                  rng.randint(2, 5)))
        return _case("", kind="group", L=",".join(map(str, sizes)),
                     splits=",".join("2" if s >= 44 else "1" for s in sizes),
                     chains=rng.choice([16, 40, 64, 96]), h=rng.choice([0.0, 0.05]), beta=0.2217)
    if kind == "infinite":
        N = _log_int(rng, 100, 100000)
        return _case("", kind="infinite", N=N, chains=_chains(rng, N, n_md + 1), n_md=n_md,
                     eps=eps * 30.0 / (30.0 + N ** 0.25), h=rng.choice([0.0, 0.02]), beta=rng.uniform(0.8, 1.2),
                     flip=rng.choice([0, 0, 1]))
    if kind == "dense":
        prec = rng.choice(["bf16", "bf16", "fp8"])
        return _case("", kind="dense", N=128 * rng.randint(4, 32), chains=rng.randint(64, 1024),
                     n_md=rng.randint(4, 12), eps=0.1 if prec == "fp8" else 0.15, prec=prec,
                     field=rng.choice([0.0, 0.1]), flip=rng.choice([0, 0, 1]), beta=0.5)
    if kind == "fp64":
        L = (_log_int(rng, 16, 256), _log_int(rng, 16, 256))
        return _case("", L="%d,%d" % L, chains=rng.randint(1, 8), n_md=rng.randint(4, 12), eps=0.08,
                     prec="fp64", h=rng.choice([0.0, 0.01]), beta=beta)
    X = rng.choice([32, 64, 96, 128, 256, 512, 1024, 8 * rng.randint(1, 40), 2 * rng.randint(2, 100)])
    Y = 2 * _log_int(rng, 4, 300)
    return _case("", kind="mh", L="%d,%d" % (X, Y), chains=max(1, min(_log_int(rng, 4, 512), int(2e7 / (X * Y)))),
                 n_traj=_log_int(rng, 8, 400), beta=beta, h=rng.choice([0.0, 0.02]))


# ------------------------------------------------------------------ inputs --
def _dims(case):
    return tuple(int(v) for v in case["L"].split(",")) if case["L"] else ()


def _members(case):
    """The single-handle cases that a case consists of (several for a group)."""
    if case["kind"] != "group":
        return [dict(case)]
    out = []
    for L, cs in zip(_dims(case), case["splits"].split(",")):
        n_md = int(math.floor(math.log(L ** 3)))   # unit trajectory length, as the paper
        out.append(dict(case, kind="lattice", L="%d,%d,%d" % (L, L, L), n_md=n_md, split=int(cs),
                        eps=1.0 / (n_md * math.sqrt(case["beta"]))))
    return out


def _sites(m):
    return m["N"] if m["N"] else math.prod(_dims(m))


def _betas(m):
    # the beta groups of a sweep, each with its share of the chains
    g = np.linspace(m["beta"], m["beta_hi"], 16)
    return g[np.arange(m["chains"]) * 16 // m["chains"]]


def _shift(m, betas):
    if m["kind"] == "lattice":
        return betas * 2 * len(_dims(m)) + 0.1
    if m["kind"] == "infinite":
        return np.maximum(betas, 1.0)
    return 2.1 * betas + 0.1   # above the semicircle edge 2 of the SK couplings


def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + what) & 0x7fffffff)
    return g


def _couplings(m, seed):
    n = m["N"]
    a = torch.randn((n, n), generator=_gen(seed, 11), device="cuda", dtype=torch.float64)
    a = torch.triu(a / math.sqrt(n), 1)
    return a + a.T


def _field(m, seed):
    if not m["field"]:
        return None
    return m["field"] * torch.randn(_sites(m), generator=_gen(seed, 12), device="cuda",
                                    dtype=torch.float64)


def _dress(m, b, xi):
    """A^(-1/2) xi for chains b, b + 1, ..."""
    betas = _betas(m)
    col = lambda v: torch.from_numpy(v[b:b + len(xi)]).cuda().float()  # noqa: E731
    beta, C = col(betas), col(_shift(m, betas))
    if m["kind"] == "dense":
        return xi / C.sqrt()[:, None]
    if m["kind"] == "infinite":
        mean = xi.mean(1, keepdim=True)
        return (xi - mean) / C.sqrt()[:, None] + mean / (C + beta).sqrt()[:, None]
    L = _dims(m)[::-1]
    lam = C.view(-1, *[1] * len(L)).expand(-1, *L[:-1], L[-1] // 2 + 1).clone()
    for d, n in enumerate(L):
        k = torch.cos(2 * math.pi * torch.arange(lam.shape[d + 1], device="cuda") / n) * 2
        lam += (beta[:, None] * k).view(-1, *[n_ if i == d else 1 for i, n_ in enumerate(lam.shape[1:])])
    f = torch.fft.rfftn(xi.view(-1, *L), dim=tuple(range(1, len(L) + 1)))
    return torch.fft.irfftn(f / lam.sqrt(), s=L, dim=tuple(range(1, len(L) + 1))).reshape(xi.shape)


def _start(m, seed, lo=0, hi=None):
    """Start configurations of chains lo..hi in the state precision: random
    spins dressed with the field's conditional law given them, s + A^(-1/2) xi
    (dense couplings: the mean of A's spectrum in place of A)."""
    hi = m["chains"] if hi is None else hi
    out = torch.empty((hi - lo, _sites(m)), device="cuda",
                      dtype=torch.float64 if m["prec"] == "fp64" else torch.float32)
    block = 64
    for b in range(lo // block * block, hi, block):   # the same values for any range asked
        g = _gen(seed, 1000 + b)
        n = min(block, m["chains"] - b)
        x = _dress(m, b, torch.randn((n, _sites(m)), generator=g, device="cuda"))
        x += torch.sign(torch.rand((n, _sites(m)), generator=g, device="cuda") - 0.5)
        a, z = max(lo, b), min(hi, b + n)
        out[a - lo:z - lo] = x[a - b:z - b].to(out.dtype)
    return out


class _State:
    """A program's handles, start configurations and their destruction."""

    def __init__(self):
        self.case, self.sims, self.psi0, self.group, self.mh = None, [], [], None, None

    def __del__(self):
        if self.group is not None:
            self.group.close()
        for s in self.sims:
            s.close()
        if self.mh is not None:
            self.mh.close()


def prepare(case, seed):
    st = _State()
    st.case, st.seed = dict(case), int(seed)
    if case["kind"] == "mh":
        dims = _dims(case)
        st.mh = pkg.IsingMH(dim=len(dims), L=dims, beta=_betas(case), h=case["h"], n_chains=case["chains"])
        r = np.random.default_rng(seed)
        n = case["chains"] * math.prod(dims)
        st.mh.set_spins(2 * (np.frombuffer(r.bytes(n), np.uint8) & 1).astype(np.int8) - 1)
        return st
    for i, m in enumerate(_members(case)):
        dims, betas = _dims(m), _betas(m)
        kw = dict(kind=m["kind"], beta=betas, C=_shift(m, betas), eps=m["eps"], n_md=m["n_md"],
                  n_chains=m["chains"], precision=PREC[m["prec"]], integrator=INTEG[m["integrator"]],
                  flip_every=m["flip"], h=m["h"])
        hv = _field(m, seed + i)
        if hv is not None:
            kw["h"] = hv.cpu().numpy()
        if m["kind"] == "lattice":
            kw.update(dim=len(dims), L=dims)
        elif m["kind"] == "dense":
            kw.update(J=_couplings(m, seed + i).cpu().numpy())
        else:
            kw.update(n_sites=m["N"])
        sim = pkg.IsingHMC(**kw)
        st.sims.append(sim)
        if m.get("split", 1) > 1:
            sim.set_chain_split(m["split"])
        psi0 = _start(m, seed + i)
        torch.cuda.synchronize()
        if m["resume"]:
            st.psi0.append(psi0)
        else:
            pkg.ising_hmc_set_state_native(sim.h, psi0.data_ptr(), 0)
        del psi0
    if case["kind"] == "group":
        st.group = pkg.IsingGroup(st.sims)
    return st


def run(state):
    case, seed = state.case, state.seed
    if state.mh is not None:
        state.mh.sweeps(case["n_traj"], seed)
        return {"spins": state.mh.spins(), "sums": state.mh.chain_sums()}
    for sim, psi0 in zip(state.sims, state.psi0):   # resumed from the checkpoint
        pkg.ising_hmc_set_state_native(sim.h, psi0.data_ptr(), 0)
    if state.group is not None:
        state.group.trajectories(case["n_traj"], seed)
    else:
        state.sims[0].trajectories(case["n_traj"], seed)
    out = []
    for sim in state.sims:
        fp64 = sim.kw["precision"] == PREC["fp64"]
        n, N = sim.kw["n_chains"], pkg.load().ising_hmc_n_sites(sim.h)
        psi = torch.empty((n, N), device="cuda", dtype=torch.float64 if fp64 else torch.float32)
        pkg.ising_hmc_get_state_native(sim.h, psi.data_ptr())
        out.append({"psi": psi, "records": sim.records()})
        if not state.psi0:
            out[-1]["sums"] = sim.chain_sums()   # running sums of the Sec. 4 estimators
    return out


def work(case):
    if case["kind"] == "mh":
        sites = case["chains"] * math.prod(_dims(case))
        # one bit per spin in, one byte out; a comparison per site and sweep
        return {"bytes": sites * 1.125, "flops": float(sites * case["n_traj"])}
    total = {"bytes": 0.0, "flops": 0.0}
    for m in _members(case):
        N, C = _sites(m), m["chains"]
        elem = 8 if m["prec"] == "fp64" else 4
        passes = (2 * m["n_md"] if m["integrator"] == "omelyan" else m["n_md"]) + 1
        # the configuration in and out, the couplings once
        total["bytes"] += 2.0 * N * C * elem + (N * N * (1 if m["prec"] == "fp8" else 2)
                                                if m["kind"] == "dense" else 0)
        if m["kind"] == "dense":
            per = 4.0 * N + 20
        elif m["kind"] == "infinite":
            per = 24.0
        else:   # two products with A, tanh, kick and drift
            per = 2 * (2 * len(_dims(m)) + 3) + 14.0
        total["flops"] += m["n_traj"] * passes * per * N * C
    return total


# ----------------------------------------------------------- FP64 statement --
_MASK = 0xffffffff


def _philox(idx, traj, chain, purpose, seed):
    """Philox4x32-10, counter (idx, traj, chain, purpose): four int64 tensors of
    32-bit values; idx and chain broadcast against each other."""
    idx, chain = torch.broadcast_tensors(idx, chain)
    c = [idx.clone(), torch.full_like(idx, traj), chain.clone(), torch.full_like(idx, purpose)]
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57   # wraps in 64 bits; both halves are kept
        c = [((p1 >> 32) & _MASK) ^ c[1] ^ k0, p1 & _MASK,
             ((p0 >> 32) & _MASK) ^ c[3] ^ k1, p0 & _MASK]
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return c


def _u23(x):
    return ((x >> 9).double() + 0.5) * 2.0 ** -23


def _u52(a, b):
    return ((a >> 6).double() * 67108864.0 + (b >> 6).double() + 0.5) * 2.0 ** -52


def _box_muller(u1, u2):
    r = torch.sqrt(-2.0 * torch.log(u1))
    return r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)


def _normals(m, n0, n1, traj, seed):
    N, per = _sites(m), 2 if m["prec"] == "fp64" else 4
    q = torch.arange((N + per - 1) // per, device="cuda")[None, :]
    c = torch.arange(n0, n1, device="cuda")[:, None]
    x = _philox(q, traj, c, 1, seed)
    if per == 2:
        z = _box_muller(_u52(x[0], x[1]), _u52(x[2], x[3]))
    else:
        z = _box_muller(_u23(x[0]), _u23(x[1])) + _box_muller(_u23(x[2]), _u23(x[3]))
    return torch.stack(z, -1).reshape(n1 - n0, -1)[:, :N]


def _uniforms(m, n0, n1, traj, seed):
    N, per = _sites(m), 2 if m["prec"] == "fp64" else 4
    q = torch.arange((N + per - 1) // per, device="cuda")[None, :]
    c = torch.arange(n0, n1, device="cuda")[:, None]
    x = _philox(q, traj, c, 3, seed)
    u = (_u52(x[0], x[1]), _u52(x[2], x[3])) if per == 2 else tuple(_u23(v) for v in x)
    return torch.stack(u, -1).reshape(n1 - n0, -1)[:, :N]


def _logu(n0, n1, traj, seed, purpose):
    c = torch.arange(n0, n1, device="cuda")
    x = _philox(torch.zeros_like(c), traj, c, purpose, seed)
    return torch.log(_u52(x[0], x[1]))


def _schedule(m):
    n = m["n_md"]
    if m["integrator"] == "leapfrog":
        return [0.5] + [1.0] * (n - 1) + [0.5], [1.0] * n + [0.0]
    lam = OMELYAN_LAMBDA
    kick = [lam]
    for s in range(n):
        kick += [1 - 2 * lam, 2 * lam if s + 1 < n else lam]
    return kick, [0.5] * (2 * n) + [0.0]


class _Exact:
    """Chains n0..n1 of a single-handle case in FP64."""

    def __init__(self, m, n0, n1, J, hv, seed):
        self.m, self.n0, self.n1, self.J, self.seed = m, n0, n1, J, seed
        col = lambda v: torch.from_numpy(np.ascontiguousarray(v[n0:n1])).cuda()[:, None]  # noqa: E731
        self.beta = col(_betas(m))
        self.C = col(_shift(m, _betas(m)))
        self.hp = self.beta * (hv[None, :] if hv is not None else m["h"])
        self.low = lambda x: x
        self.Jlow = J
        if m["prec"] == "bf16":
            self.low = lambda x: x.float().bfloat16().double()
            self.Jlow = self.low(J)
        elif m["prec"] == "fp8":
            e4m3 = lambda x: x.float().clamp(-448, 448).to(torch.float8_e4m3fn).double()  # noqa: E731
            row = (J.abs().amax(1, keepdim=True) / 448).float().double()
            self.low = lambda x: e4m3(x * 14.0) / 14.0   # operands in units of 32/448
            self.Jlow = row * e4m3(J / row)

    def apply(self, x, force=False):
        """A x; in a force of the tensor-core forms the operands of the product
        with J are the rounded ones that those forms are defined by."""
        m = self.m
        if m["kind"] == "dense":
            k = self.low(x) @ self.Jlow.T if force else x @ self.J
        elif m["kind"] == "infinite":
            k = (x.sum(1, keepdim=True) - x) / m["N"]
        else:
            v = x.view(x.shape[0], *reversed(_dims(m)))
            k = torch.zeros_like(v)
            for d in range(1, v.dim()):
                k += torch.roll(v, 1, d)
                k += torch.roll(v, -1, d)
            k = k.view(x.shape)
        return self.beta * k + self.C * x

    def evaluate(self, x, traj, seed):
        """S and the estimator values (m, E, |m| of a spin draw, |mean t|)."""
        a = self.apply(x)
        y = a + self.hp
        S = (0.5 * x * a - (y.abs() + torch.log1p(torch.exp(-2 * y.abs())))).sum(1)
        t = torch.tanh(y)
        N = x.shape[1]
        mag = t.mean(1)
        E = 0.5 * self.C[:, 0] - 0.5 * (a * t).sum(1) / N - (self.hp * t).sum(1) / N
        u = _uniforms(self.m, self.n0, self.n1, traj, seed)
        spin = torch.where(u < (1 + t) * 0.5, 1.0, -1.0).double().sum(1).abs() / N
        return S, mag, E, spin

    def trajectories(self, x, n):
        m, eps = self.m, self.m["eps"]
        kick, drift = _schedule(m)
        S, *obs = self.evaluate(x, 0xffffffff, 0)
        sums = torch.zeros((x.shape[0], 10), device="cuda", dtype=torch.float64)
        rec = torch.zeros((x.shape[0], 8), device="cuda", dtype=torch.float64)
        for traj in range(n):
            p = _normals(m, self.n0, self.n1, traj, self.seed)
            K0 = 0.5 * (p * p).sum(1)
            y = x.clone()
            for k, d in zip(kick, drift):
                p += k * eps * self.apply(torch.tanh(self.apply(y, True) + self.hp) - y, True)
                if d:
                    y += d * eps * p
            K1 = 0.5 * (p * p).sum(1)
            S1, *new = self.evaluate(y, traj, self.seed)
            dH = (K1 + S1) - (K0 + S)
            lu = _logu(self.n0, self.n1, traj, self.seed, 2)
            acc = lu < -dH
            rec = torch.stack([dH, lu, acc.double(), K0, S, K1, S1, torch.zeros_like(dH)], 1)
            x = torch.where(acc[:, None], y, x)
            S = torch.where(acc, S1, S)
            obs = [torch.where(acc, b, a) for a, b in zip(obs, new)]
            if m["flip"] and (traj + 1) % m["flip"] == 0:
                S2, *new = self.evaluate(-x, traj, self.seed)
                fl = _logu(self.n0, self.n1, traj, self.seed, 4) < -(S2 - S)
                rec[:, 7] = fl.double()
                x = torch.where(fl[:, None], -x, x)
                S = torch.where(fl, S2, S)
                obs = [torch.where(fl, b, a) for a, b in zip(obs, new)]
            mag, E, spin = obs
            sums += torch.stack([torch.ones_like(E), rec[:, 2], mag, mag * mag, E, E * E, spin,
                                 spin * spin, dH, torch.exp(-dH)], 1)
        return x, rec, sums


def exact(case, seed):
    if case["kind"] == "mh":
        return None   # integer spins and decisions: nothing is rounded
    out = []
    for i, m in enumerate(_members(case)):
        J = _couplings(m, seed + i) if m["kind"] == "dense" else None
        hv = _field(m, seed + i)
        N, C = _sites(m), m["chains"]
        psi = torch.empty((C, N), device="cuda", dtype=torch.float64)
        rec, sums = np.zeros((C, 8)), np.zeros((C, 10))
        step = max(1, min(C, int(1.2e8 / N)))
        for a in range(0, C, step):
            b = min(C, a + step)
            x = _start(m, seed + i, a, b).double()
            x, r, s = _Exact(m, a, b, J, hv, seed).trajectories(x, m["n_traj"])
            psi[a:b] = x
            rec[a:b], sums[a:b] = r.cpu().numpy(), s.cpu().numpy()
        out.append({"psi": psi, "records": rec})
        if not m["resume"]:
            out[-1]["sums"] = sums
    return out
