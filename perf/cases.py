"""What a user of this framework has it do, as timed cases.

A pass steps a simulation some collisions on and reads the result, the way a
simulation program does: `Box.step(k)` or `Batch.step(k)`, then the particles
(on the device or on the host), the observables or a velocity profile.  The
boxes, densities and options are those of the named workloads in
`paper_1801_10187_gb300/inputs.py`, of the benchmark and of the tests.  States
start in equilibrium (uniform positions, Maxwell-Boltzmann velocities; chains
as random walks), so a later pass on the same state is a pass of the same kind.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1801_10187_gb300 as mpcd

DT, KT, MASS, ALPHA = 0.1, 1.0, 1.0, 130.0  # the benchmark fluid
BEAD_MASS, BOND_K, BOND_R0, LJ_SIGMA = 5.0, 1000.0, 0.5, 0.5


def _case(name, n, rho, steps, read, **kw):
    c = {"name": name, "nx": n[0], "ny": n[1], "nz": n[2], "rho": rho, "steps": steps, "read": read,
         "precision": "mixed", "rule": "srd", "thermostat": False, "angular": False, "walls": False,
         "chains": 0, "chain_len": 0, "substeps": 0, "wca": False, "boxes": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a coupled program that looks at the particles after every collision
        _case("each-step-16c-mixed", (16, 16, 16), 10, 1, "device"),
        # the smallest box of the named workloads, in double precision, sampled now and then
        _case("tiny-10c-fp64", (10, 10, 10), 5, 100, "device", precision="fp64"),
        # a short job on host arrays: state in, thermostatted run, state out
        _case("job-32c-mixed", (32, 32, 32), 10, 300, "job", thermostat=True),
        # the paper's benchmark fluid, 10^7 particles, both precision models
        _case("fluid-100c-mixed", (100, 100, 100), 10, 25, "device"),
        _case("fluid-100c-fp64", (100, 100, 100), 10, 10, "device", precision="fp64"),
        # the Andersen rule on a ragged box
        _case("andersen-ragged-mixed", (101, 67, 89), 10, 15, "device", rule="at"),
        # angular-momentum conservation with the thermostat
        _case("angular-64c-mixed", (64, 64, 64), 10, 25, "device", thermostat=True, angular=True),
        # Poiseuille flow between walls, with the profile a viscosity fit reads
        _case("poiseuille-50x20-mixed", (50, 50, 20), 10, 25, "profile", thermostat=True, walls=True),
        # the paper's polymer benchmark: repelling chains in the double-precision solvent
        _case("polymer-50c-fp64", (50, 50, 50), 10, 4, "host", precision="fp64", chains=1024,
              chain_len=50, substeps=50, wca=True),
        # the largest: 7.8e7 particles, 2000 chains, thermostat (the benchmark's default workload)
        _case("solute-250c-mixed", (250, 250, 250), 5, 20, "device", thermostat=True, chains=2000,
              chain_len=50, substeps=10),
        # an ensemble of independent small boxes of mixed sizes, stepped together
        _case("ensemble-12-mixed", (10, 32, 0), 0, 400, "batch", boxes=12),
        # thermodynamic monitoring of a thermostatted run
        _case("monitor-100c-mixed", (100, 100, 100), 5, 10, "observables", thermostat=True),
    ]


def _edges(rng, lo, hi):
    """Three cell counts around one log-uniform edge, ragged more often than not."""
    e = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 0.3:
        return (round(e),) * 3
    return tuple(max(lo, min(hi, round(e * rng.uniform(0.75, 1.3)))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["each", "fluid", "fluid", "fp64", "job", "at", "angular", "walls", "polymer",
                       "solute", "batch", "monitor"])
    rho = rng.choice([5, 5, 10, 10, 7, 20, rng.randint(3, 30)])
    if kind == "each":
        c = _case("", _edges(rng, 8, 48), rho, 1, "device", thermostat=rng.random() < 0.5)
    elif kind == "fluid":
        c = _case("", _edges(rng, 12, 140), rho, rng.randint(5, 40), "device", thermostat=rng.random() < 0.5)
    elif kind == "fp64":
        c = _case("", _edges(rng, 8, 100), rho, rng.randint(5, 30), "device", precision="fp64",
                  thermostat=rng.random() < 0.5)
    elif kind == "job":
        c = _case("", _edges(rng, 10, 56), rho, rng.randint(100, 500), "job", thermostat=rng.random() < 0.5)
    elif kind == "at":
        c = _case("", _edges(rng, 12, 100), rho, rng.randint(5, 20), "device", rule="at")
    elif kind == "angular":
        c = _case("", _edges(rng, 12, 80), rho, rng.randint(5, 25), "device", angular=True,
                  thermostat=rng.random() < 0.5)
    elif kind == "walls":
        n = _edges(rng, 16, 80)
        c = _case("", (n[0], n[1], rng.randint(10, 40)), rho, rng.randint(10, 30), "profile", walls=True,
                  thermostat=True)
    elif kind == "polymer":
        c = _case("", _edges(rng, 20, 50), rng.choice([5, 10]), rng.randint(2, 4), "host", precision="fp64",
                  chains=1, chain_len=rng.choice([20, 50]), substeps=50, wca=True)
        c["chains"] = max(1, int(0.4 * c["nx"] * c["ny"] * c["nz"] * rng.uniform(0.4, 1.0) / c["chain_len"]))
    elif kind == "solute":
        c = _case("", _edges(rng, 40, 160), 5, rng.randint(5, 20), "device", thermostat=rng.random() < 0.7,
                  chains=rng.randint(40, 1000), chain_len=rng.choice([20, 50]), substeps=10)
    elif kind == "batch":
        lo = rng.randint(8, 16)
        c = _case("", (lo, rng.randint(lo + 4, 36), 0), 0, rng.randint(100, 400), "batch", boxes=rng.randint(4, 16))
    else:
        c = _case("", _edges(rng, 24, 100), rho, 10, "observables", thermostat=rng.random() < 0.5)
    if c["read"] != "batch":  # no more particle-steps than the largest listed case
        c["steps"] = max(1, min(c["steps"], int(1e9 / _count(c))))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _n(c):
    return c["nx"], c["ny"], c["nz"]


def _count(c):
    return int(c["rho"]) * c["nx"] * c["ny"] * c["nz"]


def _ensemble(c, seed):
    """(edge, density, angle, seed) of each box of a batch; the sizes do not depend on the seed."""
    rng = np.random.default_rng(1000 * c["boxes"] + 50 * c["nx"] + c["ny"])
    edges = rng.integers(c["nx"], c["ny"] + 1, c["boxes"])
    dens = rng.choice([5, 10], c["boxes"])
    angles = rng.choice([90.0, 120.0, 130.0], c["boxes"])
    return [(int(e), int(d), float(a), 4096 * seed + i) for i, (e, d, a) in enumerate(zip(edges, dens, angles))]


def _solvent(c, seed):
    """Uniform positions and zero-momentum Maxwell-Boltzmann velocities on the device."""
    g = torch.Generator("cuda").manual_seed(seed)
    real = torch.float32 if c["precision"] == "mixed" else torch.float64
    N = _count(c)
    pos = torch.empty((N, 3), dtype=real, device="cuda")
    for k, L in enumerate(_n(c)):
        x = torch.rand(N, dtype=torch.float64, device="cuda", generator=g).mul_(L).to(real)
        top = torch.tensor(float(L), dtype=real)
        pos[:, k] = x.clamp_(max=float(torch.nextafter(top, torch.zeros_like(top))))
    vel = torch.randn((N, 3), dtype=torch.float32, device="cuda", generator=g).to(torch.float64)
    vel.mul_(math.sqrt(KT / MASS)).sub_(vel.mean(0))
    return pos, vel.to(real)


def _unit(m, g):
    d = torch.randn((m, 3), dtype=torch.float64, device="cuda", generator=g)
    return d / d.norm(dim=1, keepdim=True)


def _chains(c, seed):
    """Chains as random walks of step r0; with the repulsion, no two beads closer than 0.9 sigma."""
    g = torch.Generator("cuda").manual_seed(seed + 77)
    L = torch.tensor(_n(c), dtype=torch.float64, device="cuda")
    m, ln = c["chains"], c["chain_len"]
    pos = torch.empty((m, ln, 3), dtype=torch.float64, device="cuda")

    def apart(p, others):
        """Which of the points p keep their distance from all the others."""
        ok = torch.ones(p.shape[0], dtype=torch.bool, device="cuda")
        if others.shape[0]:
            q = others.float()
            for i in range(0, p.shape[0], 256):
                d = p[i:i + 256, None, :].float() - q[None, :, :]
                d -= L.float() * torch.round(d / L.float())
                ok[i:i + 256] = (d * d).sum(-1).amin(1) >= (0.9 * LJ_SIGMA) ** 2
        return ok

    done = torch.zeros(m, dtype=torch.bool, device="cuda")
    for restart in range(100):  # chains that found no room start again elsewhere
        grow = torch.nonzero(~done)[:, 0]
        for j in range(ln):
            todo = grow
            for attempt in range(30):
                t = todo.numel()
                if j == 0:
                    p = torch.rand((t, 3), dtype=torch.float64, device="cuda", generator=g) * L
                else:
                    p = torch.remainder(pos[todo, j - 1] + BOND_R0 * _unit(t, g), L)
                pos[todo, j] = p
                if not c["wca"]:
                    todo = todo[:0]
                    break
                set_now = torch.ones(m, dtype=torch.bool, device="cuda")
                set_now[todo] = False
                set_now &= torch.isin(torch.arange(m, device="cuda"), grow)
                good = apart(p, torch.cat([pos[done].reshape(-1, 3), pos[grow, :j].reshape(-1, 3), pos[set_now, j]]))
                # of two beads proposed together and too close, the second tries again
                d = p[:, None, :] - p[None, :, :]
                d -= L * torch.round(d / L)
                good &= ~torch.tril((d * d).sum(-1) < (0.9 * LJ_SIGMA) ** 2, diagonal=-1).any(1)
                todo = todo[~good]
                if todo.numel() == 0:
                    break
            if todo.numel():
                grow = grow[~torch.isin(grow, todo)]
        done[grow] = True
        if bool(done.all()):
            break
    else:
        raise ValueError("no room for the chains")
    pos = pos.reshape(-1, 3)
    pos = torch.where(pos >= L, torch.zeros_like(pos), pos)
    vel = torch.randn(pos.shape, dtype=torch.float64, device="cuda", generator=g) * math.sqrt(KT / BEAD_MASS)
    return pos, vel - vel.mean(0)


def _params(c, seed):
    kw = dict(n=_n(c), dt=DT, alpha_deg=ALPHA, kT=KT, mass=MASS, seed=seed, thermostat=c["thermostat"],
              precision=c["precision"], collision=c["rule"], angular=c["angular"])
    if c["walls"]:
        kw.update(walls_z=True, body_force=(0.005, 0.0, 0.0), virt_density=float(c["rho"]))
    if c["chains"]:
        kw.update(chain_len=c["chain_len"], md_substeps=c["substeps"], solute_mass=BEAD_MASS,
                  bond_k=BOND_K, bond_r0=BOND_R0)
        if c["wca"]:
            kw.update(lj_epsilon=KT, lj_sigma=LJ_SIGMA)
    return kw


def prepare(case, seed):
    s = {"case": case}
    if case["read"] == "batch":
        b = s["batch"] = mpcd.Batch(precision=case["precision"])
        s["slots"] = [b.add_thermal(d * e ** 3, init_seed=sd, n=(e, e, e), dt=DT, kT=KT, alpha_deg=a, seed=sd)
                      for e, d, a, sd in _ensemble(case, seed)]
        b.step(0)
        return s
    box = s["box"] = mpcd.Box(**_params(case, seed))
    pos, vel = _solvent(case, seed)
    torch.cuda.synchronize()
    if case["read"] == "job":
        s["pos"], s["vel"] = (x.double().cpu().numpy() for x in (pos, vel))
    elif case["chains"]:
        sp, sv = _chains(case, seed)
        box.set_state(*(x.double().cpu().numpy() for x in (pos, vel, sp, sv)))
    else:
        box.set_state_device(pos, vel)
    if case["read"] in ("device", "profile"):
        s["out"] = (torch.empty_like(pos), torch.empty_like(vel))
        torch.cuda.synchronize()
    return s


def _beads(box):
    """The beads alone: a solute program reads them without the solvent (mpcd_get_state)."""
    out = [np.empty((box.n_solute, 3)) for _ in range(2)]
    p = [a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in out]
    rc = mpcd.lib().mpcd_get_state(box._ctx, None, None, p[0], p[1], None)
    if rc != mpcd.MPCD_OK:
        raise RuntimeError(mpcd.lib().mpcd_last_error())
    return out


def run(s):
    c = s["case"]
    if c["read"] == "batch":
        s["batch"].step(c["steps"])
        return [s["batch"].get_state(k)[:2] for k in s["slots"]]
    box = s["box"]
    if c["read"] == "job":
        box.set_state(s["pos"], s["vel"])
        box.step(c["steps"])
        return box.get_state()[:2]
    box.step(c["steps"])
    if c["read"] == "observables":
        o = box.observables()
        # not P: conserved at zero, what it shows of a run is rounding alone
        return {k: o[k] for k in ("KE", "T_kin", "T_cell_mean", "n", "occupied_cells")}
    if c["read"] == "host":
        return box.get_state()[:4]
    box.get_state_device(*s["out"])
    if c["read"] == "profile":
        return [*s["out"], box.profile(2 * c["nz"])]
    return [*s["out"], *_beads(box)] if c["chains"] else list(s["out"])


def work(case):
    """A collision step reads and writes position and velocity of every particle once, and does 48
    operations for it (cell sum, relative velocity, rotation, stream, shift); the Andersen rule and
    the angular correction do about twice that; a bead's MD substep takes about 100."""
    size = 4 if case["precision"] == "mixed" else 8
    N = sum(d * e ** 3 for e, d, _, _ in _ensemble(case, 1)) if case["read"] == "batch" else _count(case)
    per = 48 * (2 if case["rule"] == "at" or case["angular"] else 1)
    beads = case["chains"] * case["chain_len"]
    out = {"job": 96, "batch": 48, "host": 48}.get(case["read"], 0)  # host arrays in and out
    return {"bytes": case["steps"] * (N * 12 * size + beads * 96) + out * N,
            "flops": case["steps"] * (N * per + beads * case["substeps"] * 100)}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c0, c1, t, seed, purpose):
    """Philox4x32-10 of counter (c0, c1, t) under (seed, purpose); c0, c1: int64 tensors."""
    x = [c0, c1, torch.full_like(c0, t & _M32), torch.full_like(c0, t >> 32)]
    k0, k1 = seed & _M32, (seed >> 32) ^ purpose
    for _ in range(10):
        a, b = 0xD2511F53 * x[0], 0xCD9E8D57 * x[2]
        x = [((b >> 32) & _M32) ^ x[1] ^ k0, b & _M32, ((a >> 32) & _M32) ^ x[3] ^ k1, a & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return x


def _unit53(hi, lo):
    return ((hi << 21) | (lo >> 11)).double() * 2.0 ** -53


def _gamma(cell, nc, t, seed):
    """Gamma(3 (nc - 1) / 2, kT) by Marsaglia and Tsang, attempt by attempt."""
    d = 1.5 * (nc - 1).double() - 1.0 / 3.0
    cc = 1.0 / torch.sqrt(9.0 * d)
    out, todo = torch.zeros_like(d), torch.arange(d.numel(), device=d.device)
    for j in range(64):
        c = cell[todo]
        wa = _philox(c, torch.full_like(c, 1 + 2 * j), t, seed, 0x54484D4F)
        wb = _philox(c, torch.full_like(c, 2 + 2 * j), t, seed, 0x54484D4F)
        u1, u2, u3 = (_unit53(wa[i], wb[i]) for i in (0, 2, 1))
        x = torch.sqrt(-2.0 * torch.log(1.0 - u1)) * torch.cos(2.0 * math.pi * u2)
        dd, t1 = d[todo], 1.0 + cc[todo] * x
        v = t1 ** 3
        ok = (t1 > 0) & (torch.log(u3) < 0.5 * x * x + dd - dd * v + dd * torch.log(v.clamp(min=1e-300)))
        out[todo[ok]] = (dd * v * KT)[ok]
        todo = todo[~ok]
        if todo.numel() == 0:
            break
    return out


def _bonded(r, L, ln):
    d = (r.view(-1, ln, 3)[:, 1:] - r.view(-1, ln, 3)[:, :-1])
    d = d - L * torch.round(d / L)
    dist = d.norm(dim=2, keepdim=True)
    f = BOND_K * (dist - BOND_R0) / dist * d
    F = torch.zeros_like(r).view(-1, ln, 3)
    F[:, :-1] += f
    F[:, 1:] -= f
    return F.view(-1, 3)


def _pairs(r, L):
    """Every ordered pair of beads within the cutoff plus what two beads can move in a step."""
    reach, found = (2 ** (1 / 6) * LJ_SIGMA + 0.8) ** 2, []
    for i0 in range(0, r.shape[0], 512):
        d = r[i0:i0 + 512, None, :].float() - r[None, :, :].float()
        d -= L.float() * torch.round(d / L.float())
        i, j = torch.nonzero((d * d).sum(-1) < reach, as_tuple=True)
        keep = i + i0 != j
        found.append(torch.stack([i[keep] + i0, j[keep]]))
    return torch.cat(found, 1)


def _md(c, r, v, L):
    h = DT / c["substeps"]
    hh = 0.5 * h / BEAD_MASS
    ij = _pairs(r, L) if c["wca"] else None

    def force():
        F = _bonded(r, L, c["chain_len"])
        if c["wca"]:
            d = r[ij[1]] - r[ij[0]]
            d = d - L * torch.round(d / L)
            r2 = (d * d).sum(1, keepdim=True)
            x6 = (LJ_SIGMA ** 2 / r2) ** 3
            g = torch.where(r2 < 2 ** (1 / 3) * LJ_SIGMA ** 2, 24.0 * KT * x6 * (2.0 * x6 - 1.0) / r2, 0.0)
            F.index_add_(0, ij[0], -g * d)
        return F

    F = force()
    for _ in range(c["substeps"]):
        v = v + hh * F
        r = torch.remainder(r + h * v, L)
        F = force()
        v = v + hh * F
    return r, v


def _step(c, seed, t, r, v, sp, sv):
    n = torch.tensor(_n(c), device=r.device)
    L = n.double()
    if sp.shape[0]:
        sp, sv = _md(c, sp, sv, L)
    one = torch.full((1,), _M32, dtype=torch.int64, device=r.device)
    w = _philox(one, torch.zeros_like(one), t, seed, 0x53484654)
    shift = torch.stack([x.double()[0] for x in w[:3]]) * 2.0 ** -32 - 0.5
    r = torch.remainder(r + DT * v, L)
    x, y = torch.cat([r, sp]), torch.cat([v, sv])
    cell = torch.remainder(torch.floor(x - shift).long(), n)
    cell = cell[:, 0] + n[0] * (cell[:, 1] + n[1] * cell[:, 2])
    m = torch.full((x.shape[0], 1), MASS, dtype=torch.float64, device=r.device)
    m[r.shape[0]:] = BEAD_MASS
    C = int(n.prod())
    zero = torch.zeros((C, 3), dtype=torch.float64, device=r.device)
    M = torch.zeros((C, 1), dtype=torch.float64, device=r.device).index_add_(0, cell, m)
    u = zero.clone().index_add_(0, cell, m * y) / M.clamp(min=1e-300)
    ids = torch.arange(C, device=r.device)
    w = _philox(ids, torch.zeros_like(ids), t, seed, 0x524F5441)
    a = w[0].double() * 2.0 ** -32
    rad, phi = 2.0 * torch.sqrt(a * (1.0 - a)), 2.0 * math.pi * (w[1].double() * 2.0 ** -32)
    axis = torch.stack([rad * torch.cos(phi), rad * torch.sin(phi), 2.0 * a - 1.0], 1)
    d, ax = y - u[cell], axis[cell]
    al = math.radians(ALPHA)
    rot = d * math.cos(al) + torch.linalg.cross(ax, d) * math.sin(al) + ax * (ax * d).sum(1, keepdim=True) * (1.0 - math.cos(al))
    if c["thermostat"]:
        E = torch.zeros((C, 1), dtype=torch.float64, device=r.device).index_add_(0, cell, 0.5 * m * (d * d).sum(1, keepdim=True))[:, 0]
        nc = torch.bincount(cell, minlength=C)
        on = (nc >= 2) & (E > 0)
        xi = torch.ones_like(E)
        xi[on] = torch.sqrt(_gamma(ids[on], nc[on], t, seed) / E[on])
        rot = rot * xi[cell][:, None]
    y = u[cell] + rot
    N = r.shape[0]
    return r, y[:N], sp, y[N:]


def exact(case, seed):
    """SRD and its thermostat, with or without chains, in double.  A trajectory of float particles
    has no such value after a few steps: one particle that rounding puts beyond a cell face changes
    the whole of two cells, and each of their members does so again; so the mixed model's runs are
    given for two steps at most.  Observables of a longer run do not follow from the input either."""
    plain = case["rule"] == "srd" and not (case["angular"] or case["walls"])
    few = case["steps"] <= (2 if case["precision"] == "mixed" else 200)
    if not plain or not few or case["read"] in ("batch", "job", "observables"):
        return None
    pos, vel = (x.double() for x in _solvent(case, seed))
    sp, sv = _chains(case, seed) if case["chains"] else (pos[:0], vel[:0])
    for t in range(case["steps"]):
        pos, vel, sp, sv = _step(case, seed, t, pos, vel, sp, sv)
    return [pos, vel, sp, sv] if case["chains"] else [pos, vel]
