"""The work users have this library do, as cases that can be timed.

Every case goes through the Python binding (hpf.System, hpf.Batch,
hpf.Propagator) as a simulation script does: inputs are loaded once
(``prepare``), a pass advances the system or the network and reads its result
back into device tensors (``run``).  Sizes are those of the workloads in
workloads.py, of bench.py's options and of the tests; ``draw`` spreads over the
same ranges.  ``exact`` restates the method in 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1310_2041_gb300 import hpf, learned

RHO0 = 3.0
SCALE = 100.0  # the inverse size of a one-step density change
BOND, R0 = 4.0, 0.7
CHI3 = ((0.0, 1.2, 0.3), (1.2, 0.0, 0.8), (0.3, 0.8, 0.0))


# ------------------------------------------------------------------ the cases

def _melt(name, **kw):
    c = dict(kind="melt", chains=1000, len_a=5, len_b=5, solvent=0, species=2, mx=15, my=15,
             mz=15, chi=1.0, inv_kappa=0.1, every=1, steps=20, dt=0.01, thermostat=0, angle_k=0.0,
             dihedral_k=0.0, observe=False)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    cube = lambda m: dict(mx=m, my=m, mz=m)  # noqa: E731
    return [
        # a small melt, field refreshed every step, energies logged: latency and launches count
        _melt("melt_10k_every_step", observe=True),
        # the reference workload: 1M-bead diblock melt, field every 10 steps, frames of 20 steps
        _melt("melt_1m", chains=50000, len_a=10, len_b=10, chi=0.5, every=10, **cube(70)),
        # the same melt with the field refreshed every step (the accurate schedule)
        _melt("melt_1m_every_step", chains=50000, len_a=10, len_b=10, chi=0.5, steps=10, **cube(70)),
        # the largest workload: an A20 / B20 / solvent blend of 8.1M beads, three species
        _melt("blend_8m", chains=364500, len_a=20, len_b=0, solvent=810000, species=3, every=5,
              inv_kappa=0.05, **cube(140)),
        # deterministic canonical sampling of the 1M melt (every step couples all beads)
        _melt("nose_hoover_1m", chains=50000, len_a=10, len_b=10, chi=0.5, every=10, thermostat=1,
              **cube(70)),
        # semiflexible chains: angles and dihedrals on an odd mesh, energies logged
        _melt("semiflexible_200k", chains=10000, len_a=8, len_b=12, every=5, dt=0.005, angle_k=8.0,
              dihedral_k=0.5, observe=True, mx=41, my=41, mz=40),
        # chains longer than a warp segment, a ragged anisotropic mesh, Andersen collisions
        _melt("long_chains_160k", chains=1600, len_a=50, len_b=50, every=4, thermostat=2, mx=35,
              my=38, mz=41),
        # a parameter scan: 64 melts of uneven size advanced together
        dict(name="replicas_64", kind="replicas", replicas=64, min_chains=1000, max_chains=5000,
             sizes=43, len_a=8, len_b=12, every=10, steps=100),
        # an external driver: every frame's state from pinned host memory, one step, observables back
        dict(name="host_frames_1m", kind="frames", chains=50000, len_a=10, len_b=10, mx=70, my=70,
             mz=70, every=10, frames=4),
        # the density propagator: one prediction, one training step on the 1M melt's mesh
        dict(name="net_forward_70", kind="forward", mx=70, my=70, mz=70),
        dict(name="net_train_70", kind="train", mx=70, my=70, mz=70),
        # a learned window: prediction, 20 steps on the interpolated field, the judge
        dict(name="learned_window_1m", kind="learned", chains=50000, len_a=10, len_b=10, mx=70,
             my=70, mz=70, window=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, beads):
    """A mesh of about one node per unit volume, its axes a few per cent apart."""
    m = (beads / RHO0) ** (1.0 / 3.0)
    return {a: max(4, int(round(m * rng.uniform(0.93, 1.08)))) for a in ("mx", "my", "mz")}


def draw(rng):
    kind = rng.choice(["melt", "melt", "melt", "nose_hoover", "semiflexible", "long", "replicas",
                       "frames", "forward", "train", "learned"])
    if kind in ("forward", "train"):
        return dict(kind=kind, **{a: rng.randint(16, 80) for a in ("mx", "my", "mz")})
    if kind == "replicas":
        lo = rng.randint(200, 1500)
        return dict(kind="replicas", replicas=rng.randint(2, 64), min_chains=lo,
                    max_chains=lo * rng.randint(1, 3) + rng.randint(0, 99),
                    sizes=rng.randint(0, 9999), len_a=rng.randint(2, 12), len_b=rng.randint(2, 12),
                    every=rng.choice([5, 10, 20]), steps=100)
    la, lb = rng.randint(2, 32), rng.randint(2, 32)
    if kind == "long":
        la, lb = rng.randint(33, 150), rng.randint(33, 150)
    top = {"melt": 2e6, "long": 6e5, "semiflexible": 1e6, "learned": 1.2e6}.get(kind, 1.5e6)
    chains = max(1, _log(rng, 8e3, top) // (la + lb))
    beads = chains * (la + lb)
    if kind in ("frames", "learned"):
        c = dict(kind=kind, chains=chains, len_a=la, len_b=lb, **_mesh(rng, beads))
        return dict(c, window=rng.randint(8, 30)) if kind == "learned" else dict(c, every=10, frames=4)
    c = dict(chains=chains, len_a=la, len_b=lb, chi=round(rng.uniform(0.2, 2.0), 3),
             every=rng.choice([1, 2, 5, 10]), thermostat=rng.choice([0, 0, 2]),
             observe=rng.random() < 0.3)
    if kind == "melt" and rng.random() < 0.3:
        solvent = rng.randint(0, beads // 5)
        beads += solvent
        c.update(species=3, solvent=solvent)
    if kind == "semiflexible":
        c.update(angle_k=8.0, dihedral_k=rng.choice([0.0, 0.5]), dt=0.005)
    if kind == "nose_hoover":
        c.update(thermostat=1)
    return _melt(None, **c, **_mesh(rng, beads))


# ------------------------------------------------------------------ inputs

def _beads(c):
    return c["chains"] * (c["len_a"] + c["len_b"]) + c.get("solvent", 0)


def _unit(g, n):
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _system(c, seed):
    """Parameters and the initial state (device tensors, tag order) of one melt."""
    n, L, C = _beads(c), c["len_a"] + c["len_b"], c["chains"]
    box = (n / RHO0 / (c["mx"] * c["my"] * c["mz"])) ** (1.0 / 3.0)
    box = [float(np.float32(box * c[a])) for a in ("mx", "my", "mz")]
    S = c.get("species", 2)
    chi = np.array(CHI3) if S == 3 else np.array([[0.0, c.get("chi", 1.0)], [c.get("chi", 1.0), 0.0]])
    p = dict(n_beads=n, n_species=S, mesh=(c["mx"], c["my"], c["mz"]), box=tuple(box),
             inv_kappa=c.get("inv_kappa", 0.1), chi=chi, bond_k=BOND, bond_r0=R0,
             dt=c.get("dt", 0.01), gamma=1.0, seed=seed, field_every=c.get("every", 1),
             sort_every=1000, thermostat=c.get("thermostat", 0), nh_tau=1.0,
             andersen_nu=1.0 if c.get("thermostat", 0) == 2 else 0.0,
             angle_k=c.get("angle_k", 0.0), angle_cos0=-0.5, dihedral_k=c.get("dihedral_k", 0.0),
             dihedral_n=3, dihedral_delta=0.0)
    g = torch.Generator(device="cuda").manual_seed(seed)
    size = torch.tensor(box, device="cuda", dtype=torch.float64)
    walk = torch.empty((C, L, 3), device="cuda", dtype=torch.float64)
    walk[:, 0] = torch.rand((C, 3), generator=g, device="cuda", dtype=torch.float64) * size
    stiff = c.get("angle_k", 0.0) > 0.0
    t, u = _unit(g, C), _unit(g, C)
    for k in range(1, L):
        if stiff and k > 1:  # bond angles of 100 to 140 degrees, any torsion
            a, f = torch.rand((2, C, 1), generator=g, device="cuda", dtype=torch.float64)
            th, ph = (100.0 + 40.0 * a) * (math.pi / 180.0), 2.0 * math.pi * f
            n1 = torch.linalg.cross(t, u)
            n1 = n1 / n1.norm(dim=1, keepdim=True)
            m1 = torch.linalg.cross(n1, t)
            t, u = (-torch.cos(th) * t + torch.sin(th) * (torch.cos(ph) * m1 + torch.sin(ph) * n1),
                    t)
        elif not stiff:
            t = _unit(g, C)
        r = R0 + 0.05 * torch.randn((C, 1), generator=g, device="cuda", dtype=torch.float64)
        walk[:, k] = walk[:, k - 1] + r * t
    pos, kinds = walk.reshape(-1, 3), torch.zeros((C, L), device="cuda", dtype=torch.int32)
    if S == 3:
        kinds[C // 2:] = 1  # two homopolymers in solvent
        free = torch.rand((c["solvent"], 3), generator=g, device="cuda", dtype=torch.float64) * size
        pos = torch.cat([pos, free])
        kinds = torch.cat([kinds.reshape(-1), torch.full((c["solvent"],), 2, device="cuda",
                                                         dtype=torch.int32)])
    else:
        kinds[:, c["len_a"]:] = 1
        kinds = kinds.reshape(-1)
    vel = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    vel -= vel.mean(dim=0)
    i = torch.arange(C * L, device="cuda", dtype=torch.int32).reshape(C, L)
    bonds = torch.stack([i[:, :-1], i[:, 1:]], dim=2).reshape(-1, 2).contiguous()
    return p, dict(pos=pos.float().contiguous(), vel=vel.float().contiguous(), type=kinds.contiguous(),
                   bonds=bonds)


def _load(s, d):
    torch.cuda.synchronize()
    s.set_state(d["pos"], d["vel"], d["type"], d["bonds"])


def _replica_cases(c):
    rng = np.random.default_rng(c["sizes"])
    out = []
    for r in range(c["replicas"]):
        chains = int(rng.integers(c["min_chains"], c["max_chains"] + 1))
        m = max(4, int(round((chains * (c["len_a"] + c["len_b"]) / RHO0) ** (1.0 / 3.0))))
        out.append(dict(chains=chains, len_a=c["len_a"], len_b=c["len_b"], mx=m, my=m, mz=m,
                        chi=0.2 + 1.8 * r / max(c["replicas"] - 1, 1), every=c["every"]))
    return out


def _densities(c, seed, n):
    """Two-species volume fractions as a melt has them at n consecutive steps, [n][2][Mz][My][Mx]."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (2, c["mz"], c["my"], c["mx"])
    base = 0.5 + 0.2 * torch.randn(shape, generator=g, device="cuda")
    step = 0.01 * torch.randn((n,) + shape, generator=g, device="cuda")
    return (base + step.cumsum(0)).clamp_min_(0.0).contiguous()


def _weights(seed):
    return learned.init_params(seed)


def prepare(case, seed):
    c, k = case, case["kind"]
    if k in ("forward", "train"):
        net = hpf.Propagator((c["mx"], c["my"], c["mz"]))
        net.set_weights(_weights(seed))
        net.scale = SCALE
        snaps = _densities(c, seed, 3)
        torch.cuda.synchronize()
        return dict(kind=k, net=net, snaps=snaps, out=torch.empty_like(snaps[0]),
                    w=torch.empty(net.n_params, device="cuda"))
    if k == "replicas":
        systems = [_system(r, seed + 7 * i) for i, r in enumerate(_replica_cases(c))]
        batch = hpf.Batch([hpf.make_params(**p) for p, _ in systems], stream=torch.cuda.Stream())
        for i, (_, d) in enumerate(systems):
            _load(batch.replica(i), d)
        ends = np.cumsum([p["n_beads"] for p, _ in systems]).tolist()
        pos = torch.empty((ends[-1], 3), device="cuda")
        return dict(kind=k, batch=batch, steps=c["steps"], spans=list(zip([0] + ends[:-1], ends)),
                    pos=pos, vel=torch.empty_like(pos))
    p, d = _system(c, seed)
    s = hpf.System(hpf.make_params(**p))
    _load(s, d)
    st = dict(kind=k, system=s, pos=torch.empty_like(d["pos"]), vel=torch.empty_like(d["vel"]))
    if k == "melt":
        return dict(st, steps=c["steps"], observe=c["observe"], nh=c["thermostat"] == 1)
    if k == "frames":
        return dict(st, host=[[x.cpu().pin_memory() for x in f] for f in _frames(c, d, seed)])
    net = hpf.Propagator(p["mesh"])
    net.set_weights(_weights(seed))
    net.scale = 8.0
    return dict(st, net=net, window=c["window"])


def _frames(c, d, seed):
    """The state of each frame as an external program holds it: small moves from one to the next."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    pos, out = d["pos"], []
    for _ in range(c["frames"]):
        out.append((pos, d["vel"]))
        pos = pos + 0.01 * torch.randn(pos.shape, generator=g, device="cuda")
    return out


def run(st):
    k = st["kind"]
    if k == "forward":
        return st["net"].forward(st["snaps"][:2], out=st["out"])
    if k == "train":
        st["net"].train_step(st["snaps"][:2], st["snaps"][2], 1e-3)
        return st["net"].get_weights(st["w"])
    if k == "replicas":
        st["batch"].step(st["steps"])
        for r, (a, b) in enumerate(st["spans"]):
            st["batch"].replica(r).get_state(st["pos"][a:b], st["vel"][a:b])
        return st["pos"], st["vel"]
    s = st["system"]
    if k == "frames":
        return _run_frames(s, st)
    out = {}
    if k == "learned":
        stats = s.step_learned(st["net"], 2, K=st["window"], tol=1e9)
        out["eps"] = stats["eps_last"]
    else:
        s.step(st["steps"])
        if st["observe"]:
            out["energy"] = s.energy()
        if st["nh"]:
            out["xi"], out["eta"] = s.get_thermostat()
    out["pos"], out["vel"], _ = s.get_state(st["pos"], st["vel"])
    return out


def _run_frames(s, st):
    """Frame k + 1 is uploaded and enqueued while frame k's observables come back."""
    host, energies = st["host"], []
    s.upload_state(*host[0])
    s.apply_state(0)
    s.step(1)
    s.energy_start()
    s.upload_state(*host[1])
    for k in range(len(host)):
        if k + 1 < len(host):
            s.apply_state(k + 1)
            s.step(1)
        energies.append(s.energy_finish())
        if k + 1 < len(host):
            s.energy_start()
            if k + 2 < len(host):
                s.upload_state(*host[k + 2])
    pos, vel, _ = s.get_state(st["pos"], st["vel"])
    return dict(energies=np.stack(energies), pos=pos, vel=vel)


def work(case):
    c, k = case, case["kind"]
    if k in ("forward", "train"):
        V, macs = c["mx"] * c["my"] * c["mz"], 27 * (4 * 16 + 16 * 16 + 16 * 2)
        if k == "forward":
            return dict(bytes=24 * V, flops=2 * macs * V)
        return dict(bytes=24 * V + 9538 * 4 * 6, flops=2 * (3 * macs - 27 * 4 * 16) * V)
    # a bead's state read and written (28 + 24 bytes) and its frame written (24); a
    # bead-step's field, bond, noise and integration arithmetic
    if k == "replicas":
        n, steps = c["replicas"] * (c["min_chains"] + c["max_chains"]) // 2, c["steps"]
        n *= c["len_a"] + c["len_b"]
    elif k == "frames":
        return dict(bytes=_beads(c) * (c["frames"] * 52 + 24), flops=_beads(c) * c["frames"] * 250)
    else:
        n, steps = _beads(c), c.get("steps", 0) or 2 * c["window"]
    extra = (80 if c.get("angle_k") else 0) + (150 if c.get("dihedral_k") else 0)
    return dict(bytes=76 * n, flops=n * steps * (150 + extra))


# ------------------------------------------------------------------ the method in 64 bits

def _mul32(a, b):
    """High and low words of the 64-bit product of the constant a and the words b."""
    t = a * (b & 0xFFFF)
    u = a * (b >> 16) + (t >> 16)
    return u >> 16, ((u & 0xFFFF) << 16) | (t & 0xFFFF)


def _philox(tag, step, seed, word3):
    """Philox4x32-10 (Salmon et al., 2011): counter (tag, step, 0, word3), key seed."""
    c0, c1, c2, c3 = tag, torch.full_like(tag, step), torch.zeros_like(tag), torch.full_like(tag, word3)
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, c0)
        h1, l1 = _mul32(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(2 * (c >> 9) + 1).double() * 2.0 ** -24 for c in (c0, c1, c2, c3)]


def _normals(tag, step, seed):
    u = _philox(tag, step, seed, 0)
    a, b = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    w = 2.0 * math.pi
    return torch.stack([a * torch.cos(w * u[1]), a * torch.sin(w * u[1]), b * torch.cos(w * u[3])], 1)


class _Exact:
    """Melts in 64 bits, side by side: state, fields and forces.  The melts share
    everything but mesh, box, chi and seed."""

    def __init__(self, melts):
        self.melts, self.p = melts, melts[0][0]
        join = lambda f: torch.cat([f(p, d) for p, d in melts])  # noqa: E731
        each = lambda p, v, t: torch.tensor(v, device="cuda", dtype=t).expand(p["n_beads"], -1)  # noqa: E731
        self.x, self.v = join(lambda p, d: d["pos"]).double(), join(lambda p, d: d["vel"]).double()
        self.n = self.x.shape[0]
        self.tag = join(lambda p, d: torch.arange(p["n_beads"], device="cuda"))
        self.seed = join(lambda p, d: torch.full((p["n_beads"],), p["seed"], device="cuda"))
        self.m = join(lambda p, d: each(p, p["mesh"], torch.int64))
        self.inv_h = join(lambda p, d: each(p, [m / b for m, b in zip(p["mesh"], p["box"])],
                                            torch.float64).float())
        nodes = [p["n_species"] * int(np.prod(p["mesh"])) for p, _ in melts]
        self.spans = list(zip(np.cumsum([0] + nodes).tolist(), np.cumsum(nodes).tolist()))
        first = [d["type"].long() * int(np.prod(p["mesh"])) + a
                 for (p, d), (a, _) in zip(melts, self.spans)]
        self.first = torch.cat(first)  # a bead's species' first node
        self.next = join(lambda p, d: torch.zeros(p["n_beads"], dtype=torch.bool, device="cuda")
                         .index_fill_(0, d["bonds"][:, 0].long(), True))  # bonded to i + 1
        self.field_step = None

    def _corners(self):
        """Lower node, offset inside the cell and 13-bit weight of every bead, per axis."""
        s = (self.x.float() * self.inv_h).double()
        fl = torch.floor(s)
        q = (torch.floor(s * 8192.0) - fl * 8192.0).long()
        return torch.remainder(fl.long(), self.m), s - fl, q

    def _node(self, lo, dx, dy, dz):
        x, y, z = [torch.remainder(lo[:, a] + d, self.m[:, a]) for a, d in enumerate((dx, dy, dz))]
        return self.first + (z * self.m[:, 1] + y) * self.m[:, 0] + x

    def refresh(self):
        lo, _, q = self._corners()
        D = torch.zeros(self.spans[-1][1], dtype=torch.int64, device="cuda")
        for k in range(8):
            dx, dy, dz = k & 1, (k >> 1) & 1, k >> 2
            w = [q[:, a] if d else 8192 - q[:, a] for a, d in enumerate((dx, dy, dz))]
            D.index_add_(0, self._node(lo, dx, dy, dz), w[0] * w[1] * w[2])
        self.grad, self.W = torch.empty((D.shape[0], 3), device="cuda", dtype=torch.float64), 0.0
        for (p, _), (a, b) in zip(self.melts, self.spans):
            S, kappa = p["n_species"], p["inv_kappa"]
            h = [float(l) / m for l, m in zip(p["box"], p["mesh"])]
            cell = RHO0 * h[0] * h[1] * h[2]
            phi = D[a:b].double().reshape((S,) + tuple(reversed(p["mesh"]))) * (2.0 ** -39 / cell)
            chi = torch.tensor(np.asarray(p["chi"])[:S, :S], device="cuda", dtype=torch.float64)
            V = torch.einsum("ab,bzyx->azyx", chi + kappa, phi) - kappa
            self.grad[a:b] = torch.stack([(torch.roll(V, -1, ax) - torch.roll(V, 1, ax)) / (2.0 * h[i])
                                          for i, ax in enumerate((3, 2, 1))], -1).reshape(-1, 3)
            self.W += cell * (0.5 * torch.einsum("ab,azyx,bzyx->", chi, phi, phi)
                              + 0.5 * kappa * ((phi.sum(0) - 1.0) ** 2).sum())

    def bonded(self, x):
        """Bond, angle and dihedral energy of positions x."""
        b = x[1:] - x[:-1]
        ok = self.next[:-1]
        u = BOND * ((b[ok].norm(dim=1) - R0) ** 2).sum()
        if self.p["angle_k"]:
            two = ok[:-1] & ok[1:]
            a, w = -b[:-1][two], b[1:][two]
            c = (a * w).sum(1) / (a.norm(dim=1) * w.norm(dim=1))
            u = u + self.p["angle_k"] * ((c - self.p["angle_cos0"]) ** 2).sum()
        if self.p["dihedral_k"]:
            three = ok[:-2] & ok[1:-1] & ok[2:]
            b1, b2, b3 = b[:-2][three], b[1:-1][three], b[2:][three]
            A, B = torch.linalg.cross(b1, b2), torch.linalg.cross(b2, b3)
            phi = torch.atan2(b2.norm(dim=1) * (b1 * B).sum(1), (A * B).sum(1))
            u = u + self.p["dihedral_k"] * (1.0 + torch.cos(self.p["dihedral_n"] * phi
                                                            - self.p["dihedral_delta"])).sum()
        return u

    def force(self):
        x = self.x.detach().requires_grad_(True)
        F = -torch.autograd.grad(self.bonded(x), x)[0]
        lo, f, _ = self._corners()
        for k in range(8):
            dx, dy, dz = k & 1, (k >> 1) & 1, k >> 2
            w = [f[:, a] if d else 1.0 - f[:, a] for a, d in enumerate((dx, dy, dz))]
            F -= (w[0] * w[1] * w[2])[:, None] * self.grad[self._node(lo, dx, dy, dz)]
        return F

    def at(self, step):
        """The conservative force at `step`, the field refreshed when it is due."""
        if self.field_step is None or (step % self.p["field_every"] == 0 and self.field_step != step):
            self.refresh()
            self.field_step = step
        return self.force()

    def total(self, F, step):
        """With Langevin friction and noise."""
        if self.p["thermostat"] != 0:
            return F
        return F - self.v + math.sqrt(2.0 / self.p["dt"]) * _normals(self.tag, step, self.seed)

    def redraw(self, step):
        """The beads that collide at `step` (Andersen) and their new velocities."""
        u = _philox(self.tag, step, self.seed, 1)[0]
        hit = u < float(np.float32(self.p["andersen_nu"] * self.p["dt"]))
        return hit[:, None], _normals(self.tag, step, self.seed)

    def advance(self, steps):
        dt, th = self.p["dt"], self.p["thermostat"]
        xi = eta = 0.0
        dof = 3.0 * (self.n - 1)
        for step in range(steps):
            F = self.at(step)
            if th == 1:
                vE = self.v + 0.5 * dt * F
                K, h = 0.5 * float((vE * vE).sum()), 0.5 * dt
                for _ in range(2):
                    xi += 0.5 * h * (2.0 * K / dof - 1.0)
                    s = math.exp(-xi * h)
                    K, vE, eta = K * s * s, vE * s, eta + xi * h
                    xi += 0.5 * h * (2.0 * K / dof - 1.0)
                self.v = vE + 0.5 * dt * F
            else:
                F = self.total(F, step)
                v = self.v + dt * F
                if th == 2:
                    hit, u = self.redraw(step)
                    v = torch.where(hit, u + 0.5 * dt * F, v)
                self.v = v
            self.x = self.x + dt * self.v
        return xi, eta

    def observables(self, step):
        """The six values of hpf_energy at `step`: the field in force, the density of now."""
        F = self.total(self.at(step), step)
        v = self.v + 0.5 * self.p["dt"] * F
        if self.p["thermostat"] == 2:
            hit, u = self.redraw(step)
            v = torch.where(hit, u, v)
        K, U = 0.5 * float((v * v).sum()), float(self.bonded(self.x))
        grad = self.grad
        self.refresh()
        self.grad, W = grad, float(self.W)
        return np.array([K, U, W, K + U + W, float(v.sum(0).norm()), 2.0 * K / (3.0 * self.n)])


def _conv(x, W, b):
    """out[co](n) = b[co] + sum_d sum_ci W[d][ci][co] x[ci](n + d), periodic, d z-major."""
    out = b.reshape(-1, 1, 1, 1).expand(-1, *x.shape[1:])
    for o in range(27):
        d = (o // 9 - 1, o // 3 % 3 - 1, o % 3 - 1)
        out = out + torch.einsum("ic,izyx->czyx", W[o], torch.roll(x, [-k for k in d], (1, 2, 3)))
    return out


def _net(w, x, scale):
    """The network's output (the predicted change times scale) for x [4][Mz][My][Mx]."""
    h, at = torch.cat([scale * (x[2:] - x[:2]), x[2:]]), 0
    for k, (ci, co) in enumerate(learned.CHANNELS):
        W, at = w[at:at + 27 * ci * co].reshape(27, ci, co), at + 27 * ci * co
        h, at = _conv(h, W, w[at:at + co]), at + co
        if k < 2:
            h = torch.nn.functional.silu(h)
    return h


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "learned":
        return None  # two windows through a network in 16 bits: no 64-bit value
    if k in ("forward", "train"):
        snaps = _densities(c, seed, 3).double()
        w = torch.from_numpy(_weights(seed)).cuda().double()
        x = snaps[:2].reshape(4, *snaps.shape[2:])
        if k == "forward":
            return _net(w, x, SCALE) / SCALE
        w.requires_grad_(True)
        loss = ((_net(w, x, SCALE) - SCALE * (snaps[2] - snaps[1])) ** 2).mean()
        g = torch.autograd.grad(loss, w)[0]
        return (w - 1e-3 * g / (g.abs() + 1e-8)).detach()  # Adam's first step
    if k == "replicas":
        m = _Exact([_system(r, seed + 7 * i) for i, r in enumerate(_replica_cases(c))])
        m.advance(c["steps"])
        return m.x, m.v
    p, d = _system(c, seed)
    if k == "frames":
        energies = []
        for step, (pos, vel) in enumerate(_frames(c, d, seed)):
            m = _Exact([(p, dict(d, pos=pos, vel=vel))])
            F = m.total(m.at(step), step)
            m.v = m.v + p["dt"] * F
            m.x = m.x + p["dt"] * m.v
            energies.append(m.observables(step + 1))
        return dict(energies=np.stack(energies), pos=m.x, vel=m.v)
    m, out = _Exact([(p, d)]), {}
    xi, eta = m.advance(c["steps"])
    if c["observe"]:
        out["energy"] = m.observables(c["steps"])
    if c["thermostat"] == 1:
        out["xi"], out["eta"] = xi, eta
    return dict(out, pos=m.x, vel=m.v)
