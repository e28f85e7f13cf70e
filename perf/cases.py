"""The work that programs have this framework do, as cases that can be timed and compared.

Each case is one pass of a program that computes the electrostatics of charges in a spherical
cavity: an MD or Monte Carlo code that needs potentials, energies or fields at its charges (one
cavity at a time, or many at once), a Monte Carlo driver with resident chains, the request server,
and the far field of a large system.  Sizes and parameters are those of the repository's inputs,
tests and benchmark (paper_1907_01724_gb300/inputs.py), with odd and ragged sizes among them.

The results of the FP32 path (potentials, fields, energies: values with the accuracy of FP32
sums) go into the program's FP32 state, as in a mixed-precision MD code; those of the FP64 path
stay FP64.
"""
import math

import numpy as np
import torch

from paper_1907_01724_gb300 import api, batch, inputs, server

TAU = 0.1
DY_REL = 1e-5
COULOMB_K = 1.0 / (4.0 * math.pi)


# ---------------------------------------------------------------------------------------------
# the cases

def listed():
    return [
        # one small cavity, host arrays in and out: potentials and energy of a few hundred charges,
        # where launches and latency are all there is
        _single("potential_200_host", "potential", 200, 400, 20, eps=(1.0, 80.0), ka=1.0, io="host"),
        # a cavity of a solute's size with charges crowding the interface, arrays on the device
        _single("potential_2000_shell", "potential", 2000, 1000, 20, eps=(1.0, 80.0), ka=0.5, shell=0.25),
        # a ragged size from page-locked host arrays: the step of a host-side MD code
        _single("potential_4999_pinned", "potential", 4999, 1000, 20, eps=(1.0, 80.0), ka=2.0, shell=0.25, io="pinned"),
        # the largest single-cavity configuration: a primitive-model electrolyte
        _single("potential_20000", "potential", 20000, 2000, 30, eps=(78.5, 78.5), ka=3.0),
        # an MD force step of the same electrolyte, on the MD code's own stream: fields and potentials
        # in one pass
        _single("field_20000", "field", 20000, 2000, 30, eps=(78.5, 78.5), ka=3.0),
        # the FP64 path: a program that checks or calibrates against full precision
        _single("potential_1999_fp64", "potential", 1999, 1000, 20, eps=(1.0, 80.0), ka=0.5, shell=0.25, fp64=True),
        # a handful of small cavities of uneven size at once, host arrays in and out
        _many("batch_24_host", "batch", 24, 20, 700, io="host"),
        # many cavities in one call: a parameter sweep or an ensemble of replicas
        _many("batch_512", "batch", 512, 100, 10000),
        # Metropolis steps of 64 resident chains: trial moves of all chains, then the accepted ones
        _many("moves_64", "moves", 64, 500, 50000, steps=16),
        # the request server: moves and full energies of 64 chains, all offered at once
        _many("serve_64", "serve", 64, 500, 50000, requests=1000),
        # the far field: the treecode at an odd size near its break-even, and at the paper's N
        _single("far_100003", "potential", 100003, 3196, 20, eps=(2.0, 80.0), ka=5.0, theta=0.5, order=12),
        _single("far_1000000", "potential", 1000000, 3196, 20, eps=(2.0, 80.0), ka=5.0, theta=0.5, order=12),
    ]


def _single(name, kind, n, M, p, eps, ka, shell=0.0, io="device", fp64=False, theta=0.0, order=0):
    return {"name": name, "kind": kind, "n": n, "M": M, "p": p, "eps1": eps[0], "eps2": eps[1], "kappa_a": ka,
            "shell": shell, "io": io, "fp64": fp64, "theta": theta, "order": order}


def _many(name, kind, systems, n_lo, n_hi, M=1000, p=20, io="device", steps=0, requests=0):
    return {"name": name, "kind": kind, "systems": systems, "n_lo": n_lo, "n_hi": n_hi, "M": M, "p": p, "io": io,
            "steps": steps, "requests": requests}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["potential", "potential", "potential", "field", "fp64", "batch", "batch", "moves", "serve", "far",
                       "far"])
    p = rng.randint(8, 40)
    M = 2 * _log_int(rng, 100, 2000)
    eps = rng.choice([(1.0, 80.0), (2.0, 80.0), (78.5, 78.5), (1.0, 78.5)])
    ka = round(rng.uniform(0.5, 5.0), 3)
    shell = rng.choice([0.0, 0.0, 0.25])
    io = rng.choice(["device", "device", "host", "pinned"])
    if what in ("potential", "field"):
        c = _single("", what, _log_int(rng, 100, 40000), M, p, eps, ka, shell, io if what == "potential" else "device")
    elif what == "fp64":
        c = _single("", "potential", _log_int(rng, 100, 6000), M, p, eps, ka, shell, io, fp64=True)
    elif what == "far":
        c = _single("", "potential", _log_int(rng, 20000, 900000), 2 * _log_int(rng, 500, 1598), rng.randint(12, 24), eps,
                    ka, shell, "device", theta=round(rng.uniform(0.4, 0.6), 2), order=rng.choice([8, 12, 12, 16]))
        if c["theta"] < 0.5 or c["order"] > 12:  # the costlier traversals up to a third of the largest size
            c["n"] = min(c["n"], 150000 + rng.randint(0, 150000))
    else:
        lo = _log_int(rng, 20, 600)
        hi = lo * rng.randint(2, 16)
        systems = _log_int(rng, 2, 400)
        c = _many("", what, systems, lo, hi, 2 * _log_int(rng, 200, 800), rng.randint(12, 24),
                  rng.choice(["device", "host"]) if what == "batch" else "device")
        if what == "moves":
            c["systems"] = min(systems, 64)
            c["steps"] = 2 * rng.randint(2, 12)
        if what == "serve":
            c["systems"] = min(systems, 64)
            c["requests"] = _log_int(rng, 100, 1500)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------
# inputs

def _charges(rng, n, a, shell):
    k = int(shell * n)
    xyz = np.concatenate([inputs.shell(rng, k, a, 0.05 * a), inputs.uniform_ball(rng, n - k, a)])
    return xyz[rng.permutation(n)], inputs.neutral_charges(rng, n)


def _cavity(case, seed):
    rng = np.random.default_rng([seed, 1])
    xyz, q = _charges(rng, case["n"], 1.0, case["shell"])
    return inputs.System(1.0, case["eps1"], case["eps2"], case["kappa_a"], case["p"], case["M"], xyz, q, tau=TAU)


def _sizes(case):
    """The cavities' sizes: spread over the logarithm of their range, the same for every seed."""
    k = np.arange(case["systems"])
    u = (k * 0.6180339887498949 + 0.5 / case["systems"]) % 1.0
    return np.rint(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** u).astype(np.int64)


def _cavities(case, seed):
    rng = np.random.default_rng([seed, 2])
    out = []
    for n in _sizes(case):
        a = float(rng.uniform(0.8, 1.5))
        ka = float(rng.uniform(0.5, 3.0))
        eps1 = 1.0 if rng.random() < 0.5 else 78.5
        out.append(inputs.System(a, eps1, 78.5, ka / a, case["p"], case["M"], inputs.uniform_ball(rng, int(n), a),
                                 inputs.neutral_charges(rng, int(n)), tau=TAU))
    return out


def _trial(rng, a, x):
    """A trial position: a step of at most 5 % of the radius that stays inside the cavity."""
    while True:
        y = x + inputs.uniform_ball(rng, 1, 0.05 * a)[0]
        if float(y @ y) < (a * (1.0 - 1e-9)) ** 2:
            return y


def _move_steps(case, seed, systems):
    """Monte Carlo steps: one trial move of every chain in each, about half of them accepted.  The
    second half of the steps takes the accepted moves back, so that every pass starts alike."""
    rng = np.random.default_rng([seed, 3])
    half = case["steps"] // 2
    there, back = [], []
    pos = [s.xyz.copy() for s in systems]
    for _ in range(half):
        k = np.array([rng.integers(s.n) for s in systems], dtype=np.int64)
        old = np.array([x[i] for x, i in zip(pos, k)])
        new = np.array([_trial(rng, s.a, o) for s, o in zip(systems, old)])
        yes = rng.random(len(systems)) < 0.5
        there.append((k, new, yes))
        back.append((k, np.where(yes[:, None], old, new), yes))
        for c in np.nonzero(yes)[0]:
            pos[c][k[c]] = new[c]
    return there + back[::-1]


def _requests(case, seed, systems):
    """A request stream: nine moves (half accepted) to one full energy, over chains at random; every
    chain's accepted moves are taken back by its last requests, so that every pass starts alike."""
    rng = np.random.default_rng([seed, 4])
    pos = [s.xyz.copy() for s in systems]
    rows, undo = [], []
    while len(rows) + len(undo) < case["requests"]:
        c = int(rng.integers(len(systems)))
        if rng.random() >= 0.9:
            rows.append((c, server.REQ_ENERGY, 0, 0, np.zeros(3)))
            continue
        k = int(rng.integers(systems[c].n))
        x = _trial(rng, systems[c].a, pos[c][k])
        yes = int(rng.random() < 0.5 and len(rows) + len(undo) + 2 <= case["requests"])
        rows.append((c, server.REQ_DELTA, yes, k, x))
        if yes:
            undo.append((c, server.REQ_DELTA, 1, k, pos[c][k].copy()))
            pos[c][k] = x
    rows += undo[::-1]
    reqs = np.zeros(len(rows), dtype=server.REQUEST)
    for i, (c, kind, yes, k, x) in enumerate(rows):
        reqs[i] = (0.0, c, kind, yes, 0, k, x, i)
    return reqs


def _given(x, io):
    if io == "device":
        return torch.from_numpy(np.ascontiguousarray(x)).cuda()
    if io == "pinned":
        return torch.from_numpy(np.ascontiguousarray(x)).pin_memory().numpy()
    return np.ascontiguousarray(x)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("potential", "field"):
        s = _cavity(case, seed)
        stream = torch.cuda.Stream() if kind == "field" else None
        prm = api.hsma_default_params(p=s.p, M=s.M, tau=s.tau, stream=stream,
                                      precision=api.HSMA_FP64 if case["fp64"] else api.HSMA_FP32)
        h = api.hsma_create(s.a, s.eps1, s.eps2, s.kappa, prm)
        if case["theta"] > 0:
            api.hsma_set_far_field(h, case["theta"], case["order"])
        st = {"case": case, "h": h, "stream": stream, "xyz": _given(s.xyz, case["io"]), "q": _given(s.q, case["io"])}
        if case["io"] == "device":
            st["phi"] = torch.empty(s.n, dtype=torch.float64, device="cuda")
            st["E"] = torch.empty(s.n, 3, dtype=torch.float64, device="cuda") if kind == "field" else None
        else:
            st["phi"] = _given(np.empty(s.n), case["io"])
        return st
    systems = _cavities(case, seed)
    if kind == "serve":
        srv = server.Server(systems)
        srv.hsma_server_load()
        return {"case": case, "server": srv, "requests": _requests(case, seed, systems)}
    b = batch.from_systems(systems, max_requests=len(systems))
    n, xyz, q = batch.concat(systems)
    st = {"case": case, "batch": b, "n": n, "xyz": _given(xyz, case["io"]), "q": _given(q, case["io"])}
    if kind == "moves":
        # the chains are resident: their sources are built and evaluated before the first step
        b.hsma_batch_build_sources(n, st["xyz"], st["q"])
        b.hsma_batch_energy()
        st["steps"] = _move_steps(case, seed, systems)
    else:
        st["phi"] = torch.empty(len(q), dtype=torch.float64, device="cuda") if case["io"] == "device" else np.empty(len(q))
    return st


# ---------------------------------------------------------------------------------------------
# one pass

def _fp32(x):
    return x.to(torch.float32) if isinstance(x, torch.Tensor) else np.asarray(x, dtype=np.float32)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "field":
        h = st["h"]
        with torch.cuda.stream(st["stream"]):
            api.hsma_build_sources(h, st["xyz"], st["q"])
            E = api.hsma_field(h, api.HSMA_TOTAL, out=st["E"])
            phi = api.hsma_potential(h, api.HSMA_TOTAL, out=st["phi"])
            return {"field": _fp32(E), "phi": _fp32(phi)}
    if kind == "potential":
        h = st["h"]
        api.hsma_build_sources(h, st["xyz"], st["q"])
        phi = api.hsma_potential(h, api.HSMA_TOTAL, out=st["phi"])
        keep = np.array if case["fp64"] else _fp32
        if case["io"] == "device":
            return {"phi": phi if case["fp64"] else _fp32(phi)}
        return {"phi": keep(phi), "energy": keep(api.hsma_energy(h))}
    if kind == "batch":
        b = st["batch"]
        b.hsma_batch_build_sources(st["n"], st["xyz"], st["q"])
        phi = b.hsma_batch_potential(api.HSMA_TOTAL, out=st["phi"])
        if case["io"] == "device":
            return {"phi": _fp32(phi)}
        return {"phi": _fp32(phi), "energy": _fp32(b.hsma_batch_energy())}
    if kind == "moves":
        b, chains = st["batch"], np.arange(case["systems"], dtype=np.int32)
        out = []
        for k, x, yes in st["steps"]:
            out.append(b.hsma_batch_delta_energy(chains, k, x))
            b.hsma_batch_apply_moves(chains[yes], k[yes], x[yes])
        return {"delta": _fp32(np.stack(out))}
    res = st["server"].hsma_server_run(st["requests"])
    return {"value": _fp32(res["value"]), "status": res["status"].copy()}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without

def _work_one(n, M, p, field=False, far=0):
    """Operations of one cavity.  A real/Kelvin pair: a distance (8), a reciprocal root (1) and a
    multiply-add each way (4), once for both charges; a surface point: a distance, a root, the
    monopole and the dipole (17); a field triples the sums.  Moments and the series at the grid:
    4 per term.  With the far field: the charges of the 27 nearest cells of 32 instead of all."""
    near = n * 2 * 27 * 32 / 2 + 4.0 * n * (far + 1) ** 2 if far else float(n) * n
    each = 13 + (12 if field else 0)
    return near * each + float(n) * M * (17 + (12 if field else 0)) + 4.0 * (n + M) * (p + 1) ** 2


def work(case):
    kind = case["kind"]
    if kind in ("potential", "field"):
        n = case["n"]
        out = 8 * n + (24 * n if kind == "field" else 0)
        return {"bytes": 32 * n + out, "flops": _work_one(n, case["M"], case["p"], kind == "field",
                                                          case["order"] if case["theta"] > 0 else 0)}
    ns = _sizes(case).astype(float)
    if kind == "batch":
        return {"bytes": float(40 * ns.sum()), "flops": float(sum(_work_one(n, case["M"], case["p"]) for n in ns))}
    # a trial move: two positions of one charge against every charge, image and surface point, every
    # charge against its two images, and the surface series at both positions
    move = sum(4 * n * 13 + 2 * case["M"] * (17 + 8 * case["p"]) for n in ns) / len(ns)
    if kind == "moves":
        return {"bytes": float(case["steps"] * 32 * ns.sum()), "flops": float(case["steps"] * len(ns) * move)}
    full = sum(_work_one(n, case["M"], 0) for n in ns) / len(ns)
    r = case["requests"]
    return {"bytes": float(r * 32 * ns.mean()), "flops": float(0.92 * r * move + 0.08 * r * full)}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits: the method's definition in plain torch (Sec. 2.2 - 2.4 of arXiv:1907.01724)

ROWS = 1 << 24  # values of one pair block


def _series_coefficients(p, eps, mu):
    """M_n of the truncated series (Sec. 2.2), n = 0..p, from the finite sums of k_n and its derivative."""
    out = []
    for n in range(p + 1):
        s0 = s1 = 0.0
        t = 1.0
        for l in range(n, -1, -1):
            s0 += t
            s1 += l * t
            if l:
                t *= 2.0 * mu * l / ((n + l) * (n - l + 1.0))
        S = -s0 / ((mu + 1.0) * s0 + s1)
        out.append((eps * (n + 1) * S + 1.0) / (eps * n * S - 1.0))
    return out


class _Exact:
    """One cavity: sources of the method and the sums over them, all FP64."""

    def __init__(self, s):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.s, self.kc = s, COULOMB_K / s.eps1
        self.x = torch.from_numpy(np.ascontiguousarray(s.xyz)).to(dev)
        self.q = torch.from_numpy(np.ascontiguousarray(s.q)).to(dev)
        eps, mu = s.eps1 / s.eps2, s.kappa * s.a
        self.gamma = (eps - 1.0) / (eps + 1.0)
        self.dbar = self.gamma * (1.0 - (1.0 + mu) / (1.0 + eps)) - mu / (1.0 + eps)
        self.Mn = _series_coefficients(s.p, eps, mu)
        self.R = (1.0 + s.tau) * s.a
        F2 = s.M // 2 - 1
        F1 = round(F2 * (math.sqrt(5.0) - 1.0) / 2.0)
        j = torch.arange(F2 + 1, dtype=torch.float64, device=dev)
        z = -1.0 + 2.0 * j / F2
        c = (z + torch.sin(math.pi * z) / math.pi).clamp(-1.0, 1.0)
        sn = torch.sin(torch.acos(c))
        w = 2.0 * math.pi * self.R ** 2 / F2 * (1.0 + torch.cos(math.pi * z))
        ang = torch.stack([math.pi * j * F1 / F2, math.pi + math.pi * j * F1 / F2], 1)
        self.yhat = torch.stack([sn[:, None] * torch.cos(ang), sn[:, None] * torch.sin(ang),
                                 c[:, None].expand(-1, 2)], 2).reshape(-1, 3)
        self.w = w[:, None].expand(-1, 2).reshape(-1) / (4.0 * math.pi)
        self.kx, self.kq = self._images(self.x, self.q)
        self.Q, self.D = self._surface(self.x, self.q)

    def _images(self, x, q):
        a = self.s.a
        r = x.norm(dim=1, keepdim=True)
        rK = (a * a / r)[:, 0]
        return x * (a / r) ** 2, q / a * (self.gamma * rK + self.dbar * (self.R - rK) / 2.0)

    def _surface(self, x, q):
        """Monopole and dipole strengths of the grid points from the correction series of the charges."""
        s = self.s
        Q, D = torch.zeros_like(self.w), torch.zeros_like(self.w)
        r = x.norm(dim=1)
        rK = s.a * s.a / r
        pref, c = self.kc * q / s.a, self.gamma + self.dbar * (self.R - rK) / (2.0 * rK)
        u, xh = self.R / rK, x / r[:, None]
        rows = max(1, ROWS // max(1, x.shape[0]))
        for at in range(0, s.M, rows):
            t = self.yhat[at:at + rows] @ xh.T
            P0, P1 = torch.zeros_like(t), torch.ones_like(t)
            f = pref.clone()
            for n in range(s.p + 1):
                v = P1 @ (f * (self.Mn[n] - c))
                D[at:at + rows] += v
                Q[at:at + rows] += n / self.R * v
                P0, P1 = P1, ((2 * n + 1) * t * P1 - n * P0) / (n + 1)
                f = f * u
        return Q * self.w, D * self.w

    def _pairs(self, x, y, Q, field, skip=False):
        """Sums of Q_j / |x_i - y_j| and, if asked, of Q_j (x_i - y_j) / |x_i - y_j|^3."""
        phi = torch.zeros_like(x[:, 0])
        E = torch.zeros_like(x) if field else None
        rows = max(1, ROWS // max(1, y.shape[0]))
        for at in range(0, x.shape[0], rows):
            t = x[at:at + rows]
            d = [t[:, None, k] - y[None, :, k] for k in range(3)] if field else None
            if field:
                i = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).rsqrt_()
            else:
                i = torch.zeros(t.shape[0], y.shape[0], dtype=t.dtype, device=t.device)
                for k in range(3):
                    e = t[:, None, k] - y[None, :, k]
                    i.addcmul_(e, e)
                    del e
                i.rsqrt_()
            if skip:
                m = torch.arange(t.shape[0], device=t.device)
                i[m, m + at] = 0.0
            phi[at:at + rows] = i @ Q
            if field:
                i = i * i * i * Q
                for k in range(3):
                    E[at:at + rows, k] = (i * d[k]).sum(1)
        return phi, E

    def _layer(self, x):
        """Per (target, grid point): 1/d of the monopole and the dipole's central difference without
        cancellation, 2 (R - x.yhat) / (d+ d- (d+ + d-)): x.yhat and the distances d, d-, d+."""
        xy = x @ self.yhat.T
        h = 0.5 * DY_REL * self.R

        def dist(rho):
            e = torch.zeros_like(xy)
            for k in range(3):
                v = x[:, None, k] - rho * self.yhat[None, :, k]
                e.addcmul_(v, v)
            return e.sqrt_()
        d0, dm, dp = dist(self.R), dist(self.R - h), dist(self.R + h)
        return xy, d0, dm, dp

    def reaction_surface(self, x, field=False):
        phi = torch.zeros_like(x[:, 0])
        E = torch.zeros_like(x) if field else None
        h = 0.5 * DY_REL * self.R
        rows = max(1, ROWS // 2 // self.s.M)
        for at in range(0, x.shape[0], rows):
            t = x[at:at + rows]
            xy, d0, dm, dp = self._layer(t)
            phi[at:at + rows] = (1.0 / d0) @ self.Q + (2.0 * (self.R - xy) / (dp * dm * (dp + dm))) @ self.D
            if field:
                m = self.Q / d0 ** 3
                f = self.D * 2.0 * (self.R - xy) * (dp * dp + dp * dm + dm * dm) / ((dp + dm) * dm ** 3 * dp ** 3)
                g = self.D / dm ** 3
                for k in range(3):
                    yk = self.yhat[None, :, k]
                    e = t[:, None, k]
                    E[at:at + rows, k] = (m * (e - self.R * yk) + f * (e - (self.R + h) * yk) + g * yk).sum(1)
        return phi, E

    def evaluate(self, field=False):
        pc, Ec = self._pairs(self.x, self.x, self.kc * self.q, field, skip=True)
        pk, Ek = self._pairs(self.x, self.kx, self.kc * self.kq, field)
        ps, Es = self.reaction_surface(self.x, field)
        self.phi, self.phi_rf = pc + pk + ps, pk + ps
        if field:
            self.E = Ec + Ek + Es
        self.e_total = 0.5 * float((self.q * self.phi).sum())
        self.e_rf = 0.5 * float((self.q * self.phi_rf).sum())
        return self

    # moves: the energy is a sum over pairs and, with the sums U and V of the charges at the grid
    # points, over the grid: 1/2 sum (Q U + D V)
    def hold(self):
        self.U, self.V = torch.zeros_like(self.w), torch.zeros_like(self.w)
        rows = max(1, ROWS // 2 // self.s.M)
        for at in range(0, self.x.shape[0], rows):
            u, v = self._grid(self.x[at:at + rows], self.q[at:at + rows])
            self.U += u
            self.V += v
        return self

    def _grid(self, x, q):
        xy, d0, dm, dp = self._layer(x)
        return (q[:, None] / d0).sum(0), (q[:, None] * 2.0 * (self.R - xy) / (dp * dm * (dp + dm))).sum(0)

    def _terms(self, k, x, kx, kq):
        """Energy of charge k at x (its image kq at kx) with all other charges and images."""
        i = (self.x - x).norm(dim=1).reciprocal_()
        i[k] = 0.0
        j = (self.kx - x).norm(dim=1).reciprocal_()
        j[k] = 0.0
        m = (self.x - kx).norm(dim=1).reciprocal_()
        m[k] = 0.0
        qk = self.q[k]
        e = qk * (i @ self.q) + 0.5 * (qk * (j @ self.kq) + kq * (m @ self.q) + qk * kq / (x - kx).norm())
        return self.kc * e

    def move(self, k, x_new, commit):
        xo, xn = self.x[k:k + 1], torch.from_numpy(np.ascontiguousarray(x_new)).to(self.x).reshape(1, 3)
        qk = self.q[k:k + 1]
        kxn, kqn = self._images(xn, qk)
        pair = self._terms(k, xn[0], kxn[0], kqn[0]) - self._terms(k, xo[0], self.kx[k], self.kq[k])
        Qn, Dn = self._surface(xn, qk)
        Qo, Do = self._surface(xo, qk)
        Un, Vn = self._grid(xn, qk)
        Uo, Vo = self._grid(xo, qk)
        dQ, dD, dU, dV = Qn - Qo, Dn - Do, Un - Uo, Vn - Vo
        surf = 0.5 * ((dQ * self.U).sum() + ((self.Q + dQ) * dU).sum() + (dD * self.V).sum() + ((self.D + dD) * dV).sum())
        if commit:
            self.x[k], self.kx[k], self.kq[k] = xn[0], kxn[0], kqn[0]
            self.Q, self.D, self.U, self.V = self.Q + dQ, self.D + dD, self.U + dU, self.V + dV
        return pair + surf


MOST_PAIRS = 6e10  # beyond this the FP64 sums take too long


def exact(case, seed):
    kind = case["kind"]
    if kind in ("potential", "field"):
        if 2.0 * case["n"] ** 2 > MOST_PAIRS:
            return None
        e = _Exact(_cavity(case, seed)).evaluate(kind == "field")
        if kind == "field":
            return {"field": e.E, "phi": e.phi}
        return {"phi": e.phi} if case["io"] == "device" else {"phi": e.phi, "energy": np.array([e.e_total, e.e_rf])}
    systems = _cavities(case, seed)
    if 2.0 * float((_sizes(case).astype(float) ** 2).sum()) > MOST_PAIRS:
        return None
    if kind == "batch":
        each = [_Exact(s).evaluate() for s in systems]
        out = {"phi": torch.cat([e.phi for e in each])}
        if case["io"] != "device":
            out["energy"] = np.array([[e.e_total for e in each], [e.e_rf for e in each]])
        return out
    held = [_Exact(s).hold() for s in systems]
    if kind == "moves":
        return {"delta": torch.stack([torch.stack([held[c].move(int(k[c]), x[c], bool(yes[c])) for c in range(len(held))])
                                      for k, x, yes in _move_steps(case, seed, systems)])}
    energy = [e.evaluate().e_total for e in held]
    value = []
    for r in _requests(case, seed, systems):
        c = int(r["chain"])
        if r["kind"] == server.REQ_ENERGY:
            value.append(torch.as_tensor(energy[c], dtype=torch.float64, device=held[c].x.device).reshape(()))
            continue
        de = held[c].move(int(r["k"]), r["x"], bool(r["accept"]))
        if r["accept"]:
            energy[c] = energy[c] + de
        value.append(de)
    return {"value": torch.stack(value), "status": None}
