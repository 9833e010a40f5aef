"""Performance cases of the LBM-LES channel solver: what a user has it do, at the sizes users run.

Every case is a call sequence of a user's program through the package's public
entry points (``lbm.Channel``, ``lbm.Batch`` and the ``lbm_*`` functions):

  run         advance n steps, read density, velocity and wall stress on the device
  sample      advance n steps with fused plane statistics every k steps, read them
  monitor     advance n steps, then the conservation check and the allocation-free
              plane profile (what a long run does between its output times)
  checkpoint  advance n steps, save the populations to host memory, restore them
  batch       advance an ensemble of independent channels, read every member

The channels follow the recipe of the paper's turbulent channel runs
(centreline velocity 0.04, log-law profile plus 10% seeded noise, friction
velocity, viscosity and body force from Re_tau).
"""
import math

import numpy as np
import torch

from paper_2009_04352_gb300 import lbm, workload

BB, WFB, FREESLIP, NODE = 0, 1, 2, 3
RE = (180.0, 395.0, 640.0, 1000.0, 2003.0)


def _case(kind="run", nx=64, ny=32, nz=32, re=640.0, tau=0.0, wall=WFB, law=0, half=False, aa=False, mrt=False,
          steps=32, every=0, members=0, scale=0, pick=0, **name):
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, re=re, tau=tau, wall=wall, law=law, half=half, aa=aa, mrt=mrt,
                steps=steps, every=every, members=members, scale=scale, pick=pick, **name)


def listed():
    return [
        # the small channel of parity runs and examples: 100 steps, in L2, launch and latency count
        _case(name="small_fp32", tau=0.52, steps=100),
        # a Re_tau 640 production channel, whose two lattices are a little larger than L2
        _case(name="mid_fp32", nx=256, ny=64, nz=128, steps=32),
        # the largest single channel, FP32 and FP16 storage
        _case(name="large_fp32", nx=1024, ny=256, nz=512, re=2003.0, steps=16),
        _case(name="large_fp16", nx=1024, ny=256, nz=512, re=2003.0, half=True, steps=16),
        # half the memory twice over: one FP16 lattice updated in place
        _case(name="inplace_fp16", nx=512, ny=128, nz=256, re=2003.0, half=True, aa=True, steps=32),
        # the paper's collision operator (MRT + van Driest) in FP16 storage
        _case(name="mrt_fp16", nx=512, ny=128, nz=256, re=2003.0, half=True, mrt=True, steps=32),
        # the paper's A40 grid with its operator, mean profiles sampled every 10 steps
        _case("sample", name="study_mrt_sampled", nx=252, ny=80, nz=126, mrt=True, steps=100, every=10),
        # a grid of odd counts with plain bounce-back walls (the paper's reference boundary)
        _case(name="odd_fp32_bb", nx=255, ny=65, nz=127, wall=BB, steps=32),
        # save and restore of a production channel
        _case("checkpoint", name="checkpoint_fp32", nx=256, ny=64, nz=128, steps=8),
        # the watchdog of a long run: mass and momentum, and the current mean profile
        _case("monitor", name="monitor_fp32", nx=512, ny=128, nz=256, re=2003.0, steps=10),
        # the parameter study: 64 uneven channels at once
        _case("batch", name="ensemble_fp16", members=64, scale=1, pick=5, half=True, steps=16),
        # the same with small channels, where the members' launches count
        _case("batch", name="ensemble_small_fp32", members=64, scale=4, pick=5, steps=32),
    ]


def _cost(c):
    """Cell updates of a pass."""
    cells = sum(m[0] * m[1] * m[2] for m in _members(c)) if c["kind"] == "batch" else c["nx"] * c["ny"] * c["nz"]
    return cells * max(c["steps"], 1)


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choices(("run", "sample", "monitor", "checkpoint", "batch"), (60, 12, 10, 6, 12))[0]
        half, mrt = rng.random() < 0.45, rng.random() < 0.3
        c = _case(kind, re=rng.choice(RE), half=half, mrt=mrt, steps=spread(1, 100))
        if kind == "batch":
            c.update(members=spread(2, 64), scale=rng.choice((1, 2, 4)), pick=rng.randrange(1000))
            if _cost(c) <= 2.0e9:
                return c
            continue
        c.update(nx=spread(16, 1024), ny=spread(8, 256), nz=spread(8, 512), wall=rng.choice((WFB, WFB, WFB, BB, FREESLIP, NODE)),
                 law=rng.choice((0, 0, 0, 1, 2)), aa=rng.random() < 0.3)
        # most users take round counts along x; a third takes what comes
        if rng.random() < 0.65:
            c["nx"] = max(16, c["nx"] // 16 * 16)
        if c["wall"] == NODE:
            c["aa"] = False   # wall nodes run on two lattices
        if c["wall"] == BB and mrt:
            c["wall"] = WFB   # bounce-back with the damped first layer does not stay finite in long runs
        if kind == "sample":
            c["every"] = rng.choice((1, 5, 10, 20))
        if kind == "checkpoint" and c["nx"] * c["ny"] * c["nz"] > 4e6:
            continue
        if _cost(c) <= 2.0e9:
            return c


# ---------------------------------------------------------------- the channels

def _log_law(yplus):
    yp = np.asarray(yplus, dtype=np.float64)
    return np.where(yp < 1.0, yp, np.minimum(yp, np.log(np.maximum(yp, 1.0)) / 0.41 + 5.5))


def _physics(nx, ny, nz, re, tau=0.0, wall=WFB):
    """Relaxation time, body force, friction velocity, mean profile and noise of a channel at Re_tau."""
    D = (ny - 1) / 2.0 if wall == NODE else ny / 2.0
    u_tau = 0.04 / float(_log_law(re))
    if tau <= 0.0:
        tau = 0.5 + 3.0 * u_tau * D / re
    j = np.arange(ny, dtype=np.float64)
    d = np.minimum(j, ny - 1 - j) if wall == NODE else np.minimum(j + 0.5, ny - j - 0.5)
    profile = u_tau * _log_law(re * d / D)
    return dict(tau=tau, fx=u_tau * u_tau / D, u_tau=u_tau, nu=(tau - 0.5) / 3.0, profile=profile,
                noise=float(0.1 * np.mean(profile)), dist=d)


def _members(c):
    """(nx, ny, nz, re) of an ensemble's members: heights and Reynolds numbers of a study, drawn from its seed."""
    r = np.random.RandomState(c["pick"])
    out = []
    for _ in range(c["members"]):
        ny = int(r.choice((32, 48, 64, 96, 128))) // c["scale"]
        out.append((4 * ny, ny, 2 * ny, float(r.choice(RE))))
    return out


def _channel_case(nx, ny, nz, re, p, wall, law, seed):
    return workload.ChannelCase(name="channel", nx=nx, ny=ny, nz=nz, re_tau=re, tau=p["tau"], cs=0.1,
                                force=(p["fx"], 0.0, 0.0), wall=wall, u_tau=p["u_tau"], seed=seed, wall_law=law)


def _seed(seed, i=0):
    return (int(seed) * 1000003 + 7919 * i + 1) & 0x7FFFFFFF


def prepare(case, seed):
    prec = lbm.FP16_SHIFTED if case["half"] else lbm.FP32
    coll = lbm.COLLISION_MRT if case["mrt"] else lbm.COLLISION_BGK
    if case["kind"] == "batch":
        sizes = _members(case)
        phys = [_physics(*s) for s in sizes]
        b = lbm.Batch([_channel_case(*s, p, WFB, 0, 0) for s, p in zip(sizes, phys)], precision=prec)
        if case["mrt"]:
            b.set_les(coll, [p["u_tau"] for p in phys], 26.0)
        for i, (m, p) in enumerate(zip(b.members, phys)):
            m.init_channel(p["profile"], p["noise"], _seed(seed, i))
        # density and velocity of all members, one after the other
        cells = b.cells
        return dict(case=case, batch=b, rho=torch.empty(cells, device="cuda"), u=torch.empty(3 * cells, device="cuda"))
    nx, ny, nz, wall = case["nx"], case["ny"], case["nz"], case["wall"]
    p = _physics(nx, ny, nz, case["re"], case["tau"], wall)
    ch = lbm.Channel.from_case(_channel_case(nx, ny, nz, case["re"], p, wall, case["law"], 0), precision=prec,
                               layout=lbm.AA if case["aa"] else lbm.PULL2)
    if case["mrt"]:
        ch.set_les(coll, p["u_tau"], 26.0)
    ch.init_channel(p["profile"], p["noise"], _seed(seed))
    if case["kind"] == "sample":
        ch.set_stats_every(case["every"])
    return dict(case=case, ch=ch, tau=torch.empty((2, nz, nx, 2), device="cuda"),
                profile=torch.empty((ny, lbm.K_STATS), dtype=torch.float64, device="cuda"))


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b, at = state["batch"], 0
        b.step(case["steps"])
        for m in b.members:
            lbm.lbm_moments(m.handle, state["rho"][at:].data_ptr(), state["u"][3 * at:].data_ptr(), 1)
            at += m.n
        return {"rho": state["rho"], "u": state["u"]}
    ch = state["ch"]
    ch.step(case["steps"])
    if case["kind"] == "checkpoint":
        f = ch.populations()
        ch.set_populations(f)
        rho, u = ch.moments(device=True)
        return {"f": f, "rho": rho, "u": u}
    if case["kind"] == "sample":
        planes, walls, n = ch.plane_stats(reset=True)
        rho, u = ch.moments(device=True)
        return {"planes": planes, "walls": walls, "samples": n, "rho": rho, "u": u}
    if case["kind"] == "monitor":
        lbm.lbm_plane_profile_noalloc(ch.handle, state["profile"].data_ptr())
        total = ch.conservation()
        rho, u = ch.moments(device=True)
        return {"profile": state["profile"], "total": total, "rho": rho, "u": u}
    rho, u = ch.moments(device=True)
    lbm.lbm_wall_stress(ch.handle, state["tau"].data_ptr(), 1)
    return {"rho": rho, "u": u, "tau": state["tau"]}


def work(case):
    """A time step is the unit of the path: its state is read once and written once (19 populations
    each way at the storage width); outputs read the state once more and write what they return."""
    cells = sum(m[0] * m[1] * m[2] for m in _members(case)) if case["kind"] == "batch" else \
        case["nx"] * case["ny"] * case["nz"]
    f = 19 * (2 if case["half"] else 4)
    b = cells * (2 * f * case["steps"] + f + 16)
    if case["kind"] == "checkpoint":
        b += cells * (2 * f + 2 * 19 * 8)
    if case["kind"] == "monitor":
        b += cells * 2 * f
    return {"bytes": b, "flops": cells * (case["steps"] * (420 if case["mrt"] else 320) + 50)}


# ------------------------------------------- the same update in 64 bits, in plain torch

E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, 0, 1),
     (-1, 0, -1), (0, 1, 1), (0, -1, -1), (1, -1, 0), (-1, 1, 0), (1, 0, -1), (-1, 0, 1), (0, 1, -1), (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
OPP = [E.index((-x, -y, -z)) for x, y, z in E]
MIRROR = [E.index((x, -y, z)) for x, y, z in E]


def _basis():
    """Rows of the D3Q19 moment basis of d'Humieres et al. (2002)."""
    rows = []
    for i in range(19):
        r = []
        for x, y, z in E:
            q = x * x + y * y + z * z
            r.append([1, 19 * q - 30, (21 * q * q - 53 * q + 24) // 2, x, (5 * q - 9) * x, y, (5 * q - 9) * y, z,
                      (5 * q - 9) * z, 3 * x * x - q, (3 * q - 5) * (3 * x * x - q), y * y - z * z,
                      (3 * q - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                      (x * x - y * y) * z][i])
        rows.append(r)
    return rows


def _uniform(seed, cell3):
    """Top 53 bits of the first SplitMix64 output for the states seed ^ cell3, in [0, 1)."""
    def signed(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    def shift(v, n):   # logical shift of int64
        return (v >> n) & ((1 << (64 - n)) - 1)

    z = (cell3 ^ seed) + signed(0x9E3779B97F4A7C15)
    z = (z ^ shift(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * signed(0x94D049BB133111EB)
    z = z ^ shift(z, 31)
    return shift(z, 11).double() * 2.0 ** -53


def _dot(e, v):
    """e . v for a lattice direction; None where e = 0."""
    s = None
    for k in range(3):
        if e[k]:
            t = v[k] if e[k] > 0 else -v[k]
            s = t if s is None else s + t
    return s


class _Reference:
    """f[a][z][y][x]: what the step's gather reads, f_a(x, t)."""

    def __init__(self, nx, ny, nz, re, seed, tau=0.0, wall=WFB, law=0, mrt=False):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.shape, self.wall, self.law, self.mrt = (nz, ny, nx), wall, law, mrt
        self.p = p = _physics(nx, ny, nz, re, tau, wall)
        self.F = (p["fx"], 0.0, 0.0)
        cell3 = 3 * torch.arange(nx * ny * nz, dtype=torch.int64, device=self.dev).reshape(self.shape)
        u = [(2.0 * _uniform(seed, cell3 + c) - 1.0) * p["noise"] for c in range(3)]
        u[0] += torch.as_tensor(p["profile"], device=self.dev)[None, :, None]
        uu = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        self.f = []
        for a in range(19):
            eu = _dot(E[a], u)
            self.f.append(W[a] * ((1.0 - uu) if eu is None else 1.0 + 3.0 * eu + 4.5 * eu ** 2 - uu))
        # Smagorinsky constant per layer: C_s = 0.1, with van Driest damping (A+ = 26) under MRT
        cs = np.full(ny, 0.1)
        if mrt:
            cs = cs * (1.0 - np.exp(-p["dist"] * p["u_tau"] / p["nu"] / 26.0))
        self.cs2 = torch.as_tensor(cs ** 2, device=self.dev)[None, :, None]

    def moments(self):
        f = self.f
        rho = f[0].clone()
        j = [torch.full_like(rho, 0.5 * F) for F in self.F]
        for a in range(1, 19):
            rho += f[a]
            for k in range(3):
                if E[a][k]:
                    j[k].add_(f[a], alpha=E[a][k])
        return rho, [v.div_(rho) for v in j]

    def _uplus(self, R):
        """u+ from R = y+ u+ for the wall function of the case."""
        R = torch.clamp(R, min=1e-300)
        k, B = 0.41, 5.5
        if self.law == 2:
            return torch.where(R <= 8.3 ** (7.0 / 3.0), R.sqrt(), (8.3 * R ** (1 / 7)) ** 0.875)
        if self.law == 1:
            yc = 11.0
            for _ in range(200):
                yc = math.log(yc) / k + B
            up = torch.full_like(R, yc)
            for _ in range(60):
                up = up - (up - (R / up).log() / k - B) / (1.0 + 1.0 / (k * up))
            return torch.where(R.sqrt() <= yc, R.sqrt(), up)
        up = torch.where(R > 100.0, torch.minimum(R.sqrt(), R.log() / k + B), R.sqrt())
        for _ in range(60):
            q = k * up
            t2 = q.expm1() - q - q * q / 2
            y = up + math.exp(-k * B) * (t2 - q ** 3 / 6)
            up = up - (up * y - R) / (y + up * (1.0 + math.exp(-k * B) * k * t2))
        return up

    def _stress(self, rho, ux, uz):
        ut = (ux ** 2 + uz ** 2).sqrt()
        t = rho * (ut / self._uplus(ut / self.p["nu"])) ** 2
        safe = torch.where(ut > 0, ut, torch.ones_like(ut))
        return -ux / safe * t, -uz / safe * t

    def step(self):
        f, F, (nz, ny, nx) = self.f, self.F, self.shape
        rho, u = self.moments()
        self.sample = rho, u
        pi = {}
        for i in range(3):
            for k in range(i, 3):
                s = -rho * u[i] * u[k]
                if i == k:
                    s -= rho / 3.0
                for a in range(19):
                    if E[a][i] * E[a][k]:
                        s.add_(f[a], alpha=E[a][i] * E[a][k])
                pi[i, k] = s
        q = sum((1.0 if i == k else 2.0) * v * v for (i, k), v in pi.items()).sqrt()
        del pi, s
        tau = 0.5 * (self.p["tau"] + (self.p["tau"] ** 2 + 18.0 * math.sqrt(2.0) * self.cs2 * q / rho).sqrt())
        om = 1.0 / tau
        del q, tau
        uu = 1.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
        uF = sum(u[k] * F[k] for k in range(3))
        node = {}
        if self.wall == NODE:
            node = {y: [v[:, y].clone() for v in f] for y in (0, ny - 1)}
        # n_a = f^eq - f and the Guo term G_a before its rate factor
        neq, G = [], []
        for a in range(19):
            eu, eF = _dot(E[a], u), sum(E[a][k] * F[k] for k in range(3))
            eq = W[a] * rho * ((1.0 - uu) if eu is None else 1.0 + 3.0 * eu + 4.5 * eu ** 2 - uu)
            g = W[a] * ((3.0 * eF - 3.0 * uF) if eu is None else 3.0 * eF - 3.0 * uF + (9.0 * eF) * eu)
            if self.mrt:
                neq.append(eq - f[a])
                G.append(g)
            else:
                f[a] += om * (eq - f[a]) + (1.0 - 0.5 * om) * g
        if self.mrt:
            rate = [1.0, 1.19, 1.4, 1.0, 1.99, 1.0, 1.99, 1.0, 1.99, om, om, om, om, om, om, om, 1.98, 1.98, 1.98]
            for row, s in zip(_basis(), rate):
                m, g = torch.zeros_like(rho), torch.zeros_like(rho)
                for a in range(19):
                    if row[a]:
                        m.add_(neq[a], alpha=row[a])
                        g.add_(G[a], alpha=row[a])
                m = (s * m + (1.0 - 0.5 * s) * g) / sum(v * v for v in row)
                for a in range(19):
                    if row[a]:
                        f[a].add_(m, alpha=row[a])
        del neq, G
        # walls: tau_w and the correction carried by the populations that leave toward the wall
        out = []
        for y, s in ((0, 1), (ny - 1, -1)):
            xp, xm, zp, zm = (E.index((1, -s, 0)), E.index((-1, -s, 0)), E.index((0, -s, 1)), E.index((0, -s, -1)))
            if self.wall == WFB:
                tx, tz = self._stress(rho[:, y], u[0][:, y], u[2][:, y])
                for a, v in ((xp, tx), (xm, -tx), (zp, tz), (zm, -tz)):
                    f[a][:, y] += 0.5 * v
            elif self.wall == BB:
                tx, tz = -2.0 * (f[xp][:, y] - f[xm][:, y]), -2.0 * (f[zp][:, y] - f[zm][:, y])
            elif self.wall == NODE:
                n = y + s
                tx, tz = self._stress(rho[:, n], u[0][:, n], u[2][:, n])
                for a in range(19):
                    f[a][:, y] = node[y][OPP[a]]
                for a, v in ((xp, tx), (xm, -tx), (zp, tz), (zm, -tz)):
                    f[MIRROR[a]][:, y] = node[y][a] + 0.5 * v
            else:
                tx = tz = torch.zeros_like(rho[:, y])
            out.append(torch.stack((tx, tz), dim=-1))
        self.tau = torch.stack(out)
        # streaming, with the reflection of what would leave the channel
        new = [torch.roll(f[a], (E[a][2], E[a][1], E[a][0]), (0, 1, 2)) for a in range(19)]
        for a in range(19):
            if E[a][1]:
                y = 0 if E[a][1] > 0 else ny - 1
                if self.wall in (BB, NODE):
                    new[a][:, y] = f[OPP[a]][:, y]
                else:
                    new[a][:, y] = torch.roll(f[MIRROR[a]][:, y], (E[a][2], E[a][0]), (0, 1))
        self.f = new

    def planes(self, rho, u):
        cols = [rho, *u, u[0] ** 2, u[1] ** 2, u[2] ** 2, u[0] * u[1], rho * u[0], rho * u[1], rho * u[2]]
        return torch.stack([v.sum(dim=(0, 2)) for v in cols], dim=1)


def exact(case, seed):
    if _cost(case) > 3.0e9:   # more than some ten seconds of eager 64-bit torch
        return None
    if case["kind"] == "batch":
        rho, u = [], []
        for i, s in enumerate(_members(case)):
            r = _Reference(*s, _seed(seed, i), mrt=case["mrt"])
            for _ in range(case["steps"]):
                r.step()
            a, b = r.moments()
            rho.append(a.reshape(-1))
            u += [v.reshape(-1) for v in b]
        return {"rho": torch.cat(rho), "u": torch.cat(u)}
    r = _Reference(case["nx"], case["ny"], case["nz"], case["re"], _seed(seed), case["tau"], case["wall"], case["law"],
                   case["mrt"])
    planes, walls, n = 0.0, 0.0, 0
    for t in range(case["steps"]):
        r.step()
        if case["kind"] == "sample" and t % case["every"] == 0:
            planes = planes + r.planes(*r.sample)
            m = (r.tau ** 2).sum(-1)
            walls = walls + torch.stack((r.tau[..., 0], r.tau[..., 1], m.sqrt(), m), dim=-1).sum(dim=(1, 2))
            n += 1
    rho, u = r.moments()
    out = {"rho": rho, "u": torch.stack(u)}
    if case["kind"] == "checkpoint":
        out["f"] = torch.stack(r.f)
    elif case["kind"] == "sample":
        out.update(planes=planes, walls=walls, samples=None)
    elif case["kind"] == "monitor":
        total = [sum(float(v.sum()) for v in r.f)]
        total += [sum(E[a][k] * float(r.f[a].sum()) for a in range(19)) for k in range(3)]
        out.update(profile=r.planes(rho, u), total=torch.tensor(total, dtype=torch.float64))
    else:
        out["tau"] = r.tau
    return out
