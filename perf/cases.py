"""The work a user of this package has it do, as cases that can be timed and checked.

Every case is one call sequence through the public entry points, on a Hamiltonian of the
molecular-like form the tests use (a spread one-body spectrum plus decaying symmetric Cholesky
vectors, scaled so that one step's field matrix has norm 0.2 at dt = 0.005) with the
core-Hamiltonian determinant as trial.  The walkers are the trial with a random complex part,
weights around 1 and now and then a dead walker: what a population looks like a few dozen steps
into a run.  A pass starts from those walkers (``set_walkers`` on device buffers, as a run does
when it resumes), so every pass on a state is the same work with the same result.

Kinds:
  pair       the correlated run of a system and its ion (``pair_delta_E``), the headline use
  propagate  n steps of one system (``propagate``), phaseless or free projection
  energy     local energies and mixed estimates of the walkers (``energy``)
  ortho      one orthonormalisation pass of the walkers (``orthonormalise``)
  tangent    a step run with the forward-mode derivative along a one-body perturbation
  adjoint    the reverse-mode gradient dE/dh1 of a short run (``adjoint_run``)
  multidet   steps and local energies with a multi-determinant trial

Results of split-precision handles (walkers, weights and energies hold FP32-sized information
there) are taken as float32; FP64 handles' results stay float64.
"""
import math

import torch

import paper_1703_01545_gb300 as afq

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64, C128 = torch.float64, torch.complex128


def _case(name, kind, prec, M, X, n_up, n_dn, nw, steps=1, repeats=1, free=False, dets=0, dt=0.005):
    c = dict(kind=kind, prec=prec, M=M, X=X, n_up=n_up, n_dn=n_dn, nw=nw, steps=steps,
             repeats=repeats, free=free, dets=dets, dt=dt)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The headline run: neutral and ion at M = 128 on shared fields, two measurement blocks.
        _case("pair_split_m128", "pair", "split", 128, 768, 16, 16, 4096, 10, 11),
        # The same call on the smallest pair (the FCI-checkable one): 8 blocks of latency.
        _case("pair_fp64_m8", "pair", "fp64", 8, 24, 2, 2, 128, 40, 11, dt=0.01),
        # A medium system in split precision, where one step is a few hundred microseconds.
        _case("propagate_split_m64", "propagate", "split", 64, 320, 8, 8, 2048, 10),
        # The largest basis: V_HS and the propagator of a 200-orbital system.
        _case("propagate_split_m200", "propagate", "split", 200, 1000, 9, 9, 2048, 5),
        # Free projection at sizes nothing divides.
        _case("propagate_split_odd_free", "propagate", "split", 101, 555, 11, 10, 777, 5, free=True),
        # The default precision on the throughput workload.
        _case("propagate_fp64_m64", "propagate", "fp64", 64, 320, 8, 8, 2048, 2),
        # Measurement alone: exchange and Coulomb energy of a large and of a default population.
        _case("energy_split_m128", "energy", "split", 128, 768, 16, 16, 4096, repeats=11),
        _case("energy_fp64_m64", "energy", "fp64", 64, 320, 8, 8, 2048, repeats=11),
        # Re-orthonormalisation on resuming a large population.
        _case("ortho_split_m128", "ortho", "split", 128, 768, 16, 15, 4096),
        # Derivatives of a short run: all of dE/dh1 (reverse mode), one direction (forward mode).
        _case("adjoint_fp64_m96", "adjoint", "fp64", 96, 480, 12, 12, 128, 10),
        _case("tangent_fp64_m40", "tangent", "fp64", 40, 200, 6, 5, 300, 5, 3),
        # A truncated CI trial.
        _case("multidet_fp64_m64", "multidet", "fp64", 64, 320, 8, 8, 256, 2, dets=15),
    ]


# what a drawn case may cost at most: method operations of one pass
_MOST = {"split": 4e12, "fp64": 6e10}


def draw(rng):
    kind, prec = rng.choice([("pair", "split"), ("pair", "fp64"), ("propagate", "split"),
                             ("propagate", "split"), ("propagate", "fp64"), ("propagate", "fp64"),
                             ("energy", "split"), ("energy", "fp64"), ("ortho", "split"),
                             ("ortho", "fp64"), ("adjoint", "fp64"), ("tangent", "fp64"),
                             ("multidet", "fp64")])

    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    M = log_int(8, 128 if kind in ("adjoint", "tangent", "multidet") else 200)
    n_up = log_int(max(1, M // 16), min(20, M // 3, 4096 // (2 * M)))
    n_dn = rng.randint(max(1 if kind == "pair" else 0, n_up - 2), n_up)
    X = max(1, int(M * rng.uniform(3.0, 8.0)))
    nw = log_int(24, 4096)
    steps = {"pair": 5 * rng.randint(1, 3), "adjoint": 5 * rng.randint(1, 2)}.get(kind, rng.randint(1, 8))
    if kind in ("energy", "ortho"):
        steps = 1
    repeats = 1 if kind == "adjoint" else rng.randint(1, 11)
    free = kind == "propagate" and rng.random() < 0.25
    dets = rng.randint(2, 20) if kind == "multidet" else 0
    c = _case(None, kind, prec, M, X, n_up, n_dn, nw, steps, repeats, free, dets, rng.choice([0.005, 0.01]))
    while c["nw"] > 16 and work(c)["flops"] > _MOST[prec]:
        c["nw"] = max(16, int(c["nw"] / 1.3))
    c["repeats"] = min(c["repeats"], c["nw"])
    return c


# ---- inputs ----

def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _hamiltonian(c, seed):
    """h1 [M, M], L [X, M, M], orbitals (ascending eigenvectors of h1) on the device."""
    M, X, g = c["M"], c["X"], _generator(seed)
    i = torch.arange(M, device=DEV, dtype=F64)
    off = torch.triu(torch.randn(M, M, generator=g, device=DEV, dtype=F64), 1)
    off = off * 0.05 * torch.exp(-(i[:, None] - i[None, :]).abs() / 4)
    h1 = torch.diag(torch.linspace(-2.0, 3.0, M, device=DEV, dtype=F64)) + off + off.T
    decay = 0.3 * torch.exp(-4.0 * torch.arange(X, device=DEV, dtype=F64) / X)
    sigma = float(decay.square().sum().sqrt())
    u = torch.triu(torch.randn(X, M, M, generator=g, device=DEV, dtype=F64))
    u = u * (decay * math.sqrt(2.0) / (math.sqrt(M) * sigma))[:, None, None]
    L = u + torch.triu(u, 1).transpose(1, 2)
    orb = torch.linalg.eigh(h1.cpu())[1].to(DEV)
    return h1, L, orb


def _spin_down_of_ion(c):
    return c["n_dn"] - 1


def _walkers(c, start, seed):
    """phi [2, Nw, M, N] and w [2, Nw] in the layout of set_walkers."""
    g = _generator(seed * 7919 + 5)
    M, nw, N = c["M"], c["nw"], start.shape[1]
    noise = torch.randn(2, nw, M, N, generator=g, device=DEV, dtype=F64) * (0.3 / math.sqrt(2 * M))
    noise[0] += start
    w = torch.zeros(2, nw, device=DEV, dtype=F64)
    w[0] = 0.5 + torch.rand(nw, generator=g, device=DEV, dtype=F64)
    if nw >= 64 and not c["dets"]:
        # killed by the phaseless cut earlier in the run (the local energy of a dead walker has no
        # meaning, and with several determinants none that its frozen walker defines)
        w[0, 17::61] = 0.0
    return noise.contiguous(), w


def _determinants(c, orb):
    """dets [Nd, M, N], coefficients: the aufbau determinant and excitations of its top orbitals."""
    nu, nd, M = c["n_up"], c["n_dn"], c["M"]
    dets, coef = [], []
    for d in range(c["dets"]):
        up, dn = list(range(nu)), list(range(nd))
        if d > 0:
            a, b = d % 4, d // 4
            up[nu - 1 - min(a % 2, nu - 1)] = min(M - 1, nu + a // 2 + b)
            if nd and d % 3 == 0:
                dn[nd - 1] = min(M - 1, nd + b)
        dets.append(torch.cat([orb[:, up], orb[:, dn]], dim=1))
        coef.append(0.9 if d == 0 else 0.3 * (-1) ** d / (d + 1))
    return torch.stack(dets), torch.tensor(coef, dtype=F64, device=DEV)


def _inputs(c, seed):
    h1, L, orb = _hamiltonian(c, seed)
    nu, nd = c["n_up"], c["n_dn"]
    trial = torch.cat([orb[:, :nu], orb[:, :nd]], dim=1).contiguous()
    d = dict(h1=h1, L=L, orb=orb, trial=trial)
    g = _generator(seed * 104729 + 3)
    start = trial
    if c["dets"]:
        d["dets"], d["coef"] = _determinants(c, orb)
        # a determinant that overlaps every one of the expansion
        mix = trial + torch.randn(trial.shape, generator=g, device=DEV, dtype=F64) * (0.5 / math.sqrt(c["M"]))
        start = torch.cat([torch.linalg.qr(mix[:, :nu].cpu())[0], torch.linalg.qr(mix[:, nu:].cpu())[0]], dim=1).to(DEV)
    d["start"] = start.contiguous()
    d["phi"], d["w"] = _walkers(c, start, seed)
    if c["kind"] == "pair":
        nb = nu + _spin_down_of_ion(c)
        d["trial_B"] = trial[:, :nb].contiguous()
        d["phi_B"], d["w_B"] = d["phi"][..., :nb].contiguous(), d["w"]
    if c["kind"] == "tangent":
        p = torch.randn(c["M"], c["M"], generator=g, device=DEV, dtype=F64) * 0.1
        d["P"] = p + p.T
    d["seed"] = int(seed) % 100003 + 1
    return d


def _system(c, d, trial, n_dn):
    kw = dict(dt=c["dt"], n_walkers=c["nw"], n_repeats=c["repeats"], seed=d["seed"],
              mode=afq.FREE if c["free"] else afq.PHASELESS,
              precision=afq.BF16X3 if c["prec"] == "split" else afq.FP64)
    if c["dets"]:
        kw.update(dets=d["dets"].cpu().numpy(), coeffs=d["coef"].cpu().numpy(), start=d["start"].cpu().numpy())
        trial = None
    else:
        trial = trial.cpu().numpy()
    return afq.System(d["h1"].cpu().numpy(), d["L"].cpu().numpy(), trial, c["n_up"], n_dn, **kw)


def prepare(case, seed):
    c, d = case, _inputs(case, seed)
    s = dict(case=c, phi=d["phi"], w=d["w"], A=_system(c, d, d["trial"], c["n_dn"]))
    if c["kind"] == "pair":
        s["B"] = _system(c, d, d["trial_B"], _spin_down_of_ion(c))
        s["phi_B"] = d["phi_B"]
    if c["kind"] == "tangent":
        s["P"] = d["P"].cpu().numpy()
    if c["kind"] == "energy":
        afq.afqmc_set_walkers(s["A"].h, d["phi"], d["w"])
    return s


def _taken(c, x):
    x = x if isinstance(x, torch.Tensor) else torch.from_numpy(x)
    if x.is_complex():
        x = torch.view_as_real(x)
    return x.float() if c["prec"] == "split" else x


def _state(c, sysm):
    """Walkers, weights and alive flags, copied out on the device."""
    phi = torch.empty(2, c["nw"], c["M"], sysm.N, device=DEV, dtype=F64)
    w = torch.empty(2, c["nw"], device=DEV, dtype=F64)
    alive = torch.empty(c["nw"], device=DEV, dtype=torch.int32)
    afq.afqmc_get_state(sysm.h, phi, None, w, alive)
    return dict(phi=_taken(c, phi), w=_taken(c, w), alive=alive)


def run(state):
    c, A = state["case"], state["A"]
    kind = c["kind"]
    if kind == "energy":
        el, em, ws = A.energy()
        return dict(e_local=_taken(c, el), e_mixed=_taken(c, em), w_sum=_taken(c, ws))
    afq.afqmc_set_walkers(A.h, state["phi"], state["w"])
    if kind == "pair":
        B = state["B"]
        afq.afqmc_set_walkers(B.h, state["phi_B"], state["w"])
        res = afq.pair_delta_E(A, B, c["steps"], energy_every=5, mgs_every=5)
        return dict(E=_taken(c, res["E"]), A=_state(c, A), B=_state(c, B))
    if kind == "adjoint":
        e, grad = A.adjoint_run(c["steps"], mgs_every=5, energy_every=5)
        return dict(e=torch.tensor(e, dtype=F64), grad=grad, A=_state(c, A))
    if kind == "tangent":
        A.set_tangent(state["P"])
        A.propagate(c["steps"])
        em, dm, de = A.energy_tangent()
        return dict(e_mixed=em, de_mixed=dm, de_local=_taken(c, de), A=_state(c, A))
    if kind == "ortho":
        A.orthonormalise()
        return _state(c, A)
    A.propagate(c["steps"])
    if kind == "multidet":
        el, em, ws = A.energy()
        return dict(e_local=_taken(c, el), e_mixed=em, w_sum=ws, A=_state(c, A))
    return _state(c, A)


# ---- what a pass cannot do without ----

def _step_flops(c, n_up, n_dn):
    M, X, N = c["M"], c["X"], n_up + n_dn
    nd = max(1, c["dets"])
    fb = 0 if c["free"] else 4 * X * N * M * nd
    vhs = 4 * (M * (M + 1) // 2) * X
    return c["nw"] * (fb + vhs + 6 * 8 * M * M * N + 2 * 4 * M * M * N
                      + nd * (4 * M * (n_up ** 2 + n_dn ** 2) + 8 * M * (n_up ** 2 + n_dn ** 2)))


def _energy_flops(c, n_up, n_dn):
    return c["nw"] * max(1, c["dets"]) * 4 * c["X"] * c["M"] * (n_up ** 2 + n_dn ** 2)


def _ortho_flops(c, n_up, n_dn):
    return c["nw"] * 8 * c["M"] * (n_up ** 2 + n_dn ** 2)


def work(case):
    c = case
    M, X, nu, nd, kind = c["M"], c["X"], c["n_up"], c["n_dn"], c["kind"]
    out = 4 if c["prec"] == "split" else 8
    f = b = 0.0
    for n_dn in ([nd, _spin_down_of_ion(c)] if kind == "pair" else [nd]):
        N = nu + n_dn
        step, en, mgs = (fn(c, nu, n_dn) for fn in (_step_flops, _energy_flops, _ortho_flops))
        walkers = c["nw"] * 2 * M * N
        b += 8 * (X * (M * (M + 1) // 2) + M * M + M * N * max(1, c["dets"]))
        b += (8 + out) * walkers
        if kind in ("pair", "adjoint"):
            blocks = c["steps"] // 5
            # the reverse sweep takes every product of the forward run twice more
            f += (c["steps"] * step + blocks * (mgs + en)) * (3 if kind == "adjoint" else 1)
        elif kind == "tangent":
            f += 2 * (c["steps"] * step + en)
        elif kind == "energy":
            f += en
        elif kind == "ortho":
            f += mgs
        else:
            f += c["steps"] * step + (en if kind == "multidet" else 0)
    if kind == "energy":
        b = 8.0 * (X * (M * (M + 1) // 2) + c["nw"] * (2 * M * (nu + nd) + 2))
    return dict(bytes=float(b), flops=float(f))


# ---- the same in plain torch, 64 bits ----

class _Exact:
    """The method of the entry points' documentation for one system, in complex128."""

    def __init__(self, c, d, trial, n_dn, h1=None):
        self.c, self.L, self.trial = c, d["L"], trial
        self.h1 = d["h1"] if h1 is None else h1
        nu = c["n_up"]
        self.spins = [(a, b) for a, b in ((0, nu), (nu, nu + n_dn)) if b > a]
        self.seed, self.dt, self.sq = d["seed"], c["dt"], math.sqrt(c["dt"])
        self.Lf = self.L.reshape(c["X"], -1)
        P = trial @ trial.T
        self.rho = self.Lf @ P.reshape(-1)
        lp = self.L.permute(1, 0, 2).reshape(c["M"], -1)
        const = -0.5 * lp @ lp.T + torch.einsum("g,gij->ij", self.rho, self.L)
        self.K = self.h1 + const
        # exp(-dt K / 2) by its series: the norm of the exponent is far below 1
        one = torch.eye(c["M"], dtype=F64, device=self.K.device)
        self.expK = one
        for k in range(24, 0, -1):
            self.expK = one + (-0.5 * self.dt / k) * (self.K @ self.expK)
        self.C = -0.5 * float(self.rho @ self.rho)
        if c["dets"]:
            self.dets, self.coef = list(d["dets"]), d["coef"]
        else:
            self.dets, self.coef = [trial], None
        det = self.h1.detach() if isinstance(self.h1, torch.Tensor) else self.h1
        self.E_T = float(self._one_energy(trial, trial[None].to(C128), det).real[0])

    def _theta(self, D, phi):
        log, th = 0, []
        for a, b in self.spins:
            O = D[:, a:b].T.to(C128) @ phi[:, :, a:b]
            sign, lad = torch.linalg.slogdet(O)
            log = log + torch.complex(lad, torch.angle(sign))
            th.append(torch.linalg.solve(O.transpose(1, 2), phi[:, :, a:b].transpose(1, 2)).transpose(1, 2))
        return log, torch.cat(th, dim=2)

    def _shares(self, phi):
        """log <psi_T|phi>, [(share_d, Theta_d)]"""
        parts = [self._theta(D, phi) for D in self.dets]
        if self.coef is None:
            return parts[0][0], [(None, parts[0][1])]
        logs = torch.stack([p[0] for p in parts])
        top = logs.real.max(dim=0).values
        t = self.coef[:, None] * torch.exp(logs - top)
        tot = t.sum(dim=0)
        return top + torch.log(tot), [(t[k] / tot, p[1]) for k, p in enumerate(parts)]

    def _real_times(self, z, R):
        return torch.complex(z.real @ R, z.imag @ R)

    def force(self, parts):
        out = 0
        for (share, th), D in zip(parts, self.dets):
            lt = (self.L @ D).permute(0, 2, 1).reshape(self.c["X"], -1)       # [g, (n, i)]
            r = self._real_times(th.transpose(1, 2).reshape(th.shape[0], -1), lt.T)
            out = out + (r if share is None else share[:, None] * r)
        return out

    def _one_energy(self, D, phi, h1=None, theta=None):
        h1 = self.h1 if h1 is None else h1
        th = self._theta(D, phi)[1] if theta is None else theta
        e = ((h1 @ D).to(C128) * th).sum(dim=(1, 2))       # tr(h1 G), G_ji = Theta_in D_jn
        lt, chunk, two = self.L @ D, max(1, int(3e7 / (self.c["X"] * 32 * 32))), []
        for w0 in range(0, th.shape[0], chunk):
            t = th[w0:w0 + chunk]
            coul, exch = 0, 0
            for a, b in self.spins:
                # T[w, g, a, b] = sum_i lt[g, i, a] Theta[w, i, b]
                la = lt[:, :, a:b].permute(0, 2, 1).reshape(-1, lt.shape[1])
                z = t[:, :, a:b].permute(1, 0, 2).reshape(lt.shape[1], -1)
                T = torch.complex(la @ z.real, la @ z.imag).reshape(self.c["X"], b - a, t.shape[0], b - a)
                coul = coul + torch.einsum("gawa->wg", T)
                exch = exch + torch.einsum("gawb,gbwa->w", T, T)
            two.append(0.5 * (coul * coul).sum(dim=1) - 0.5 * exch)
        return e + torch.cat(two)

    def energy(self, phi):
        _, parts = self._shares(phi)
        out = 0
        for (share, th), D in zip(parts, self.dets):
            e = self._one_energy(D, phi, theta=th)
            out = out + (e if share is None else share * e)
        return out

    def fields(self, t):
        """Normals of step t: Philox-4x32-10 with counter (g / 2, k, t, 0), then Box-Muller."""
        m32, nj = 0xFFFFFFFF, (self.c["X"] + 1) // 2
        dev = self.L.device
        c0 = torch.arange(nj, device=dev)[None, :].expand(self.c["nw"], nj)
        c1 = torch.arange(self.c["nw"], device=dev)[:, None].expand(self.c["nw"], nj)
        c2, c3 = torch.full_like(c0, t), torch.zeros_like(c0)
        k0, k1 = self.seed & m32, (self.seed >> 32) & m32

        def hi_lo(a, x):                        # a * x for 32-bit a, x: its two 32-bit halves
            low, high = a * (x & 0xFFFF), a * (x >> 16)
            mid = (low >> 16) + (high & m32)
            return (high >> 32 << 16) + (mid >> 16) & m32, (mid << 16 | low & 0xFFFF) & m32

        for _ in range(10):
            h0, l0 = hi_lo(0xD2511F53, c0)
            h1, l1 = hi_lo(0xCD9E8D57, c2)
            c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
            k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
        u1 = (((c1 << 21) | (c0 >> 11)) + 1).to(F64) * 2.0 ** -53
        u2 = ((c3 << 21) | (c2 >> 11)).to(F64) * 2.0 ** -53
        r = torch.sqrt(-2.0 * torch.log(u1))
        z = torch.stack([r * torch.cos(2 * math.pi * u2), r * torch.sin(2 * math.pi * u2)], dim=2)
        return z.reshape(self.c["nw"], 2 * nj)[:, :self.c["X"]]

    def step(self, phi, w, alive, t):
        """One step of every walker: (phi, w complex, alive); dead ones stay as they are."""
        M, c = self.c["M"], self.c
        x = self.fields(t)
        log0, parts = self._shares(phi)
        xbar = torch.zeros_like(x, dtype=C128)
        if not c["free"]:
            xbar = -1j * self.sq * (self.force(parts) - self.rho)
            mag = xbar.abs()
            xbar = torch.where(mag > 1.0, xbar / torch.where(mag > 1.0, mag, 1.0), xbar)
        cg = x - xbar
        log_s = -1j * self.sq * (cg @ self.rho.to(C128))
        new = []
        E = self.expK
        chunk = max(1, int(2.5e8 / (M * M)))
        for w0 in range(0, phi.shape[0], chunk):
            A = (1j * self.sq) * self._real_times(cg[w0:w0 + chunk], self.Lf).reshape(-1, M, M)
            term = acc = E.to(C128) @ phi[w0:w0 + chunk]
            for m in range(1, 7):
                term = A @ term / m
                acc = acc + term
            new.append(E.to(C128) @ acc)
        new = torch.cat(new)
        log_r = log_s + self._shares(new)[0] - log0
        log_i = log_r + (x * xbar).sum(dim=1) - 0.5 * (xbar * xbar).sum(dim=1) - self.dt * (self.C - self.E_T)
        if c["free"]:
            nw, still = w * torch.exp(log_i), alive
        else:
            f = torch.exp(log_i.real) * torch.clamp(torch.cos(log_r.imag), min=0.0)
            nw = w * f
            still = alive & (nw.real > 0)
        phi = torch.where(alive[:, None, None], new, phi)
        return phi, torch.where(still, nw, torch.zeros_like(nw)), still

    def ortho(self, phi, alive):
        q = []
        for a, b in self.spins:
            p = phi[:, :, a:b]
            low = torch.linalg.cholesky(p.mH @ p)
            q.append(torch.linalg.solve_triangular(low.mH, p, upper=True, left=False))
        return torch.where(alive[:, None, None], torch.cat(q, dim=2), phi)

    def mixed(self, w, el):
        """Per repeat: mixed estimate and weight sum."""
        R, nw = self.c["repeats"], self.c["nw"]
        grp = torch.arange(nw, device=w.device) * R // nw
        if not self.c["free"]:
            w, el = w.real, el.real
        num = torch.zeros(R, dtype=w.dtype, device=w.device).index_add(0, grp, w * el)
        den = torch.zeros(R, dtype=w.dtype, device=w.device).index_add(0, grp, w)
        return (num / den).real, den.real


def _planes(z):
    return torch.stack([z.real, z.imag])


def exact(case, seed):
    c, d = case, _inputs(case, seed)
    phi0 = torch.complex(d["phi"][0], d["phi"][1])
    w0 = torch.complex(d["w"][0], d["w"][1])
    alive0 = w0 != 0

    def out(phi, w, alive):
        return dict(phi=_planes(phi), w=_planes(w), alive=alive.to(torch.int32))

    ex = _Exact(c, d, d["trial"], c["n_dn"])
    kind = c["kind"]
    if kind == "energy":
        el = ex.energy(phi0)
        em, ws = ex.mixed(w0, el)
        return dict(e_local=torch.view_as_real(el), e_mixed=em, w_sum=ws)
    if kind == "ortho":
        return out(ex.ortho(phi0, alive0), w0, alive0)
    if kind == "pair":
        exB = _Exact(c, d, d["trial_B"], _spin_down_of_ion(c))
        phiB = torch.complex(d["phi_B"][0], d["phi_B"][1])
        st, series = [[ex, phi0, w0, alive0], [exB, phiB, w0, alive0]], []
        for t in range(c["steps"]):
            for s in st:
                s[1:] = s[0].step(*s[1:], t)
                if (t + 1) % 5 == 0:
                    s[1] = s[0].ortho(s[1], s[3])
            if (t + 1) % 5 == 0:
                series.append(torch.stack([s[0].mixed(s[2], s[0].energy(s[1]))[0] for s in st]))
        return dict(E=torch.stack(series), A=out(*st[0][1:]), B=out(*st[1][1:]))

    def whole(h1):
        """A run from h1: its walkers, and at its measurements the energies."""
        s = _Exact(c, d, d["trial"], c["n_dn"], h1)
        s.E_T = ex.E_T
        phi, w, alive, es = phi0, w0, alive0, []
        for t in range(c["steps"]):
            phi, w, alive = s.step(phi, w, alive, t)
            if kind == "adjoint" and (t + 1) % 5 == 0:
                phi = s.ortho(phi, alive)
                es.append(s.mixed(w, s.energy(phi))[0][0])
        return s, phi, w, alive, es

    if kind == "adjoint":
        h1 = d["h1"].clone().requires_grad_(True)
        _, phi, w, alive, es = whole(h1)
        e = torch.stack(es).mean()
        grad, = torch.autograd.grad(e, h1)
        return dict(e=e.detach(), grad=grad, A=out(phi.detach(), w.detach(), alive))
    if kind == "tangent":
        def measured(lam):
            s, phi, w, alive, _ = whole(d["h1"] + lam * d["P"])
            el = s.energy(phi)
            return s.mixed(w, el)[0], torch.view_as_real(el), phi, w, alive
        em, _, phi, w, alive = measured(0.0)
        h = 1e-4                       # fourth-order central difference of the whole run
        dd = [measured(k * h)[:2] for k in (-2, -1, 1, 2)]
        dm, de = ((dd[0][q] - 8 * dd[1][q] + 8 * dd[2][q] - dd[3][q]) / (12 * h) for q in (0, 1))
        return dict(e_mixed=em, de_mixed=dm, de_local=de, A=out(phi, w, alive))
    phi, w, alive = phi0, w0, alive0
    for t in range(c["steps"]):
        phi, w, alive = ex.step(phi, w, alive, t)
    if kind == "multidet":
        el = ex.energy(phi)
        em, ws = ex.mixed(w, el)
        return dict(e_local=torch.view_as_real(el), e_mixed=em, w_sum=ws, A=out(phi, w, alive))
    return out(phi, w, alive)
