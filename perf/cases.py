"""Performance cases of the ferrofluid library: what programs built on it call, at the sizes they
call it with.

A case is a dict of plain values.  `prepare` makes what such a program holds before the call (device
arrays and a context), `run` makes one pass through the public interface (`ff.py`), `work` states the
bytes and operations the pass cannot do without, and `exact` evaluates the same definitions in 64 bits
with plain torch (Barnes-Hut included: the opening decisions are the method's, taken in the case's
tree precision; every sum is formed in double).

Sizes and parameters are those of the repository's benchmark, tests and magnetisation driver: gases at
volume fraction 0.02 to 0.1, the 4096-particle dense cube, chains of 64 touching particles, batches of
dilute systems with log-uniform sizes; theta 0.5 (0.7 with the dipole-position terms), dt 1e-3.
"""
import math

import numpy as np
import torch

from paper_1212_2934_gb300 import ff

DT, INERTIA, KT, LJ_RCUT = 1e-3, 0.4, 1.0, 2.5
FLOPS = 68          # per dipole interaction (field and force)
FLOPS_QUAD = 160    # with the dipole-position terms


def listed():
    return [
        # a small ensemble's field, as an analysis script or a test asks for it: launches and latency
        dict(name="field_n1000", kind="field", n=1000, precision="f32", phi=0.05, theta=0.5,
             leaf_max=1, quad=0),
        # an ordinary field evaluation at a ragged size
        dict(name="field_n65521", kind="field", n=65521, precision="f32", phi=0.05, theta=0.5,
             leaf_max=1, quad=0),
        # the more accurate expansion at the angle it is meant for
        dict(name="field_quad_n131071", kind="field", n=131071, precision="f32", phi=0.05,
             theta=0.7, leaf_max=1, quad=1),
        # double precision, where a reference trajectory or an accuracy check is wanted
        dict(name="field_f64_n49999", kind="field", n=49999, precision="f64", phi=0.05, theta=0.5,
             leaf_max=1, quad=0),
        # the exact sum, the method's comparator
        dict(name="allpairs_n20011", kind="allpairs", n=20011, precision="f32", phi=0.05),
        # time steps: the dense cube in double precision
        dict(name="step_dense_f64", kind="step", geometry="dense", n=4096, precision="f64",
             phi=0.52, theta=0.5, leaf_max=1, steps=2),
        # time steps: the million-particle gas of the headline benchmark
        dict(name="step_n1048576", kind="step", geometry="gas", n=1048576, precision="f32",
             phi=0.05, theta=0.5, leaf_max=1, steps=2),
        # time steps: four million particles in chains, mixed precision
        dict(name="step_chains_mixed", kind="step", geometry="chains", n=4194304,
             precision="mixed", phi=0.01, theta=0.5, leaf_max=1, steps=2),
        # time steps of many dilute systems together, as the magnetisation curve is run
        dict(name="batch_64", kind="batch", nsys=64, nmin=1024, nmax=65536, precision="f32",
             phi=0.02, theta=0.5, leaf_max=1, steps=2),
        # the energy and its gradient (backward direction of the field)
        dict(name="grad_n262144", kind="grad", n=262144, precision="f32", phi=0.05, theta=0.5,
             leaf_max=1),
        # reverse mode through time steps
        dict(name="sensitivity_n50021", kind="sensitivity", n=50021, precision="f32", phi=0.05,
             theta=0.5, leaf_max=1, steps=6, every=3),
        # the allocation-free key ordering
        dict(name="order_n100003", kind="order", n=100003, phi=0.05),
    ]


def _logint(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n))


def draw(rng):
    kind = rng.choice(["field", "field", "field64", "allpairs", "step", "step", "batch", "grad",
                       "sensitivity", "order"])
    phi = round(rng.uniform(0.02, 0.1), 4)
    theta = rng.choice([0.4, 0.5, 0.5, 0.6, 0.7])
    leaf = rng.choice([1, 1, 1, 4, 8])
    if kind == "field":
        return dict(kind="field", n=_logint(rng, 700, 1048576), precision=rng.choice(["f32", "f32",
                    "mixed"]), phi=phi, theta=theta, leaf_max=leaf, quad=rng.choice([0, 0, 1]))
    if kind == "field64":
        return dict(kind="field", n=_logint(rng, 700, 80000), precision="f64", phi=phi,
                    theta=theta, leaf_max=leaf, quad=0)
    if kind == "allpairs":
        return dict(kind="allpairs", n=_logint(rng, 700, 65536),
                    precision=rng.choice(["f32", "f32", "mixed"]), phi=phi)
    if kind == "step":
        geometry = rng.choice(["gas", "gas", "chains"])
        n = _logint(rng, 2000, 1500000)
        if geometry == "chains":
            n = max(64, n // 64 * 64)
            phi = 0.01
        return dict(kind="step", geometry=geometry, n=n, precision=rng.choice(["f32", "mixed"]),
                    phi=phi, theta=theta, leaf_max=leaf, steps=2)
    if kind == "batch":
        return dict(kind="batch", nsys=_logint(rng, 3, 80), nmin=_logint(rng, 200, 2000),
                    nmax=_logint(rng, 4000, 50000), precision="f32", phi=0.02, theta=0.5,
                    leaf_max=1, steps=2)
    if kind == "grad":
        return dict(kind="grad", n=_logint(rng, 700, 300000), precision=rng.choice(["f32", "f32",
                    "mixed"]), phi=phi, theta=rng.choice([0.5, 0.6]), leaf_max=leaf)
    if kind == "sensitivity":
        return dict(kind="sensitivity", n=_logint(rng, 2000, 60000), precision="f32", phi=phi,
                    theta=0.5, leaf_max=1, steps=rng.choice([4, 6]), every=rng.choice([2, 3]))
    return dict(kind="order", n=_logint(rng, 700, 131072), phi=phi)


# ------------------------------------------------------------------ inputs
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt):
    g = torch.Generator(device=_dev())
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _unit(n, g):
    v = torch.randn((n, 3), generator=g, device=_dev(), dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _gas(n, phi, g):
    """Hard-core gas: randomly occupied sites of a cubic lattice of spacing 1.5 (1.0 above volume
    fraction 0.15), each centre moved within its site so that no two come closer than 1."""
    sp = 1.5 if phi <= 0.15 else 16.0 / 15.0
    side = (n * (math.pi / 6.0) / phi) ** (1.0 / 3.0)
    m = max(int(round(side / sp)), 1)
    while m ** 3 < n:
        m += 1
    site = torch.randperm(m ** 3, generator=g, device=_dev())[:n]
    q = torch.stack([site // (m * m), (site // m) % m, site % m], dim=1).to(torch.float64)
    jit = (sp - 1.0) / 2.0
    r = torch.rand((n, 3), generator=g, device=_dev(), dtype=torch.float64) * 2.0 - 1.0
    return (q + 0.5) * sp + r * jit, m * sp


def _chains(n, length, phi, g):
    """Straight chains of touching particles: cubic blocks, each with one main direction and a
    lattice of rods along it, randomly occupied, each rod shifted and tilted within its place."""
    nch = n // length
    pitch = (math.pi / 6.0 / phi) ** 0.5 * 0.9
    per = int((length + 2.0) // pitch)
    block = max(length + 2.0, per * pitch)
    nb = 1
    while nb ** 3 * per * per < nch:
        nb += 1
    d = _dev()
    rod = torch.randperm(nb ** 3 * per * per, generator=g, device=d)[:nch]
    b, c = rod // (per * per), rod % (per * per)
    main = torch.randint(0, 3, (nb ** 3,), generator=g, device=d)[b]
    room = (pitch - 1.5) / 2.0
    r = torch.rand((nch, 4), generator=g, device=d, dtype=torch.float64) * 2.0 - 1.0
    s0 = ((c // per).to(torch.float64) + 0.5) * pitch + r[:, 0] * room * 0.6
    s1 = ((c % per).to(torch.float64) + 0.5) * pitch + r[:, 1] * room * 0.6
    tilt = r[:, 2:4] * (0.4 * room / (0.5 * length))
    axis = torch.cat([tilt, torch.ones((nch, 1), device=d, dtype=torch.float64)], dim=1)
    axis = axis / axis.norm(dim=1, keepdim=True)
    t = torch.arange(length, device=d, dtype=torch.float64) - 0.5 * (length - 1)
    local = torch.stack([s0, s1, torch.full_like(s0, 0.5 * block)], dim=1)
    p = local[:, None, :] + t[None, :, None] * axis[:, None, :]
    roll = (torch.arange(3, device=d)[None, :] + main[:, None]) % 3
    p = torch.gather(p, 2, roll[:, None, :].expand(nch, length, 3))
    axis = torch.gather(axis, 1, roll)
    bq = torch.stack([b // (nb * nb), (b // nb) % nb, b % nb], dim=1).to(torch.float64) * block
    sign = torch.randint(0, 2, (nch, 1), generator=g, device=d).to(torch.float64) * 2.0 - 1.0
    u = (axis * sign)[:, None, :].expand(nch, length, 3)
    return (p + bq[:, None, :]).reshape(-1, 3), u.reshape(-1, 3).contiguous(), nb * block


def _sizes(case):
    k, lo, r = case["nsys"], case["nmin"], case["nmax"] / case["nmin"]
    return [int(round(lo * r ** ((i + 0.5) / k))) for i in range(k)]


def _inputs(case, seed):
    """The case's particles (tensors in the state's type) and run parameters."""
    g = _gen(seed, 17)
    dt = torch.float64 if case.get("precision") == "f64" else torch.float32
    kind = case["kind"]
    s = dict(h_ext=[0.0, 0.0, 1.0], dip_scale=1.0, gamma=0.1)
    if kind == "batch":
        parts = [_gas(m, case["phi"], g) for m in _sizes(case)]
        pos = torch.cat([p for p, _ in parts])
        s["sizes"] = np.array([p.shape[0] for p, _ in parts], dtype=np.int64)
        s["sides"] = np.array([a for _, a in parts])
        k = len(parts)
        s["fields"] = np.zeros((k, 3))
        s["fields"][:, 2] = 5.0 * ((np.arange(k) * 37) % k) / max(k - 1, 1)
        s.update(dip_scale=0.125, gamma=1.0)
        side = float(s["sides"].max())
        u = _unit(pos.shape[0], g)
    elif case.get("geometry") == "chains":
        pos, u, side = _chains(case["n"], 64, case["phi"], g)
    else:
        pos, side = _gas(case["n"], case["phi"], g)
        u = _unit(pos.shape[0], g)
        if case.get("geometry") == "dense":
            s["h_ext"] = [0.0, 0.0, 0.5]
    n = pos.shape[0]
    s["n"], s["side"] = n, side
    s["pos"], s["u"] = pos.to(dt).contiguous(), u.to(dt).contiguous()
    if kind in ("step", "batch", "sensitivity"):
        v = torch.randn((n, 3), generator=g, device=_dev(), dtype=torch.float64) * KT ** 0.5
        w = torch.randn((n, 3), generator=g, device=_dev(), dtype=torch.float64)
        s["vel"] = v.to(dt)
        s["omega"] = (w * (KT / INERTIA) ** 0.5).to(dt)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    n, kind = s["n"], case["kind"]
    s["case"] = case
    s["stream"] = torch.cuda.Stream()
    if kind == "order":
        s["keys"] = torch.empty(n, dtype=torch.int64, device="cuda")
        s["order"] = torch.empty(n, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        return s
    side = s["side"]
    p = ff.ff_params_default(
        n=n, precision=case["precision"], theta=case.get("theta", 0.5),
        leaf_max=case.get("leaf_max", 1), dt=DT, gamma_t=s["gamma"], gamma_r=s["gamma"],
        inertia=INERTIA, kT=KT, dip_scale=s["dip_scale"], lj_rcut=LJ_RCUT, h_ext=s["h_ext"],
        box_lo=(0, 0, 0), box_hi=(side, side, side), walls=1, seed=7,
        quadrupole=case.get("quad", 0), stream=s["stream"].cuda_stream)
    s["ctx"] = ff.ff_create(p)
    if kind == "batch":
        sides = s["sides"]
        ff.ff_set_systems(s["ctx"], s["sizes"], s["fields"], np.zeros((len(sides), 3)),
                          np.repeat(sides[:, None], 3, axis=1))
    if kind in ("field", "allpairs"):
        s["h"], s["f"] = torch.empty_like(s["pos"]), torch.empty_like(s["pos"])
    torch.cuda.synchronize()
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    # the library works on its own stream: after whatever made the inputs
    s["stream"].wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s["stream"]):
        if kind == "order":
            ff.ff_morton_order_noalloc(s["pos"], s["keys"], s["order"], s["stream"])
            return dict(keys=s["keys"], order=s["order"])
        ctx = s["ctx"]
        if kind in ("field", "allpairs", "grad"):
            ff.ff_set_particles(ctx, s["pos"], s["u"])
            if kind == "grad":
                dt = np.float64 if s["pos"].dtype == torch.float64 else np.float32
                e, gp, gu = ff.ff_energy_grad(ctx, ff.FF_ALGO_BH, case["theta"], dtype=dt,
                                              device_like=s["pos"])
                return dict(energy=e, grad_pos=gp, grad_u=gu)
            algo = ff.FF_ALGO_AP if kind == "allpairs" else ff.FF_ALGO_BH
            ff.ff_dipolar_field(ctx, algo, case.get("theta", 0.5), True, s["h"], s["f"])
            return dict(h=s["h"], f=s["f"])
        ff.ff_set_step(ctx, 0)
        ff.ff_set_particles(ctx, s["pos"], s["u"], s["vel"], s["omega"])
        if kind == "sensitivity":
            mz, g = ff.ff_mz_sensitivity(ctx, case["steps"], case["every"])
            return dict(mz=mz, dmz_dh=g)
        ff.ff_step(ctx, case["steps"])
        out = {}
        if kind == "batch":
            m, _ = ff.ff_system_moments(ctx, reset=True)
            out["moments"] = m
        dt = np.float64 if s["pos"].dtype == torch.float64 else np.float32
        x, u, v, w = ff.ff_get_particles(ctx, dtype=dt, device_like=s["pos"])
        out.update(pos=x, u=u, vel=v, omega=w)
        return out


def work(case):
    """Bytes: the inputs and outputs once.  Operations: the dipole interactions (field and force)
    times the operations of one.  A Barnes-Hut particle has about
    a (0.5 / theta)^2 log2(n / b) of them for volume-filling gases (866 at n = 1,048,576 and 717 at
    n = 262,144, theta = 0.5)."""
    kind = case["kind"]
    n = sum(_sizes(case)) if kind == "batch" else case["n"]
    w = 8 if case.get("precision") == "f64" else 4
    if kind == "order":
        return {"bytes": n * (12 + 12), "flops": 0}
    if kind == "allpairs":
        return {"bytes": n * 12 * w, "flops": float(n) * (n - 1) * FLOPS}

    def inter(m):
        grow = max(math.log2(max(m, 2)) - 8.4, 1.0)
        return min(m - 1, 75.0 * (0.5 / case["theta"]) ** 2 * grow)

    if kind == "batch":
        per = sum(m * inter(m) for m in _sizes(case))
    else:
        per = n * inter(n)
    if kind == "field":
        return {"bytes": n * 12 * w, "flops": per * (FLOPS_QUAD if case["quad"] else FLOPS)}
    if kind == "grad":
        return {"bytes": n * 12 * w, "flops": 2.0 * per * FLOPS}
    if kind == "sensitivity":
        return {"bytes": n * 12 * w, "flops": 3.0 * per * FLOPS * case["steps"]}
    return {"bytes": n * 24 * w, "flops": per * FLOPS * case["steps"]}


# ------------------------------------------------- the same definitions in 64 bits
def _spread(q):
    out = torch.zeros_like(q)
    for b in range(21):
        out |= ((q >> b) & 1) << (3 * b)
    return out


def _morton(pos):
    """63-bit keys of the root cube (lowest corner, largest extent), each operation rounded in the
    positions' own type; returns keys, corner, side."""
    mn = pos.min(dim=0).values
    side = (pos.max(dim=0).values - mn).max()
    if not float(side) > 0.0:
        side = torch.ones_like(side)
    q = torch.floor((pos - mn) * (torch.full_like(side, 2097152.0) / side))
    q = q.clamp(0, 2097151).to(torch.int64)
    return (_spread(q[:, 0]) << 2) | (_spread(q[:, 1]) << 1) | _spread(q[:, 2]), mn, side


def _compact(key):
    out = torch.zeros_like(key)
    for b in range(21):
        out |= ((key >> (3 * b)) & 1) << b
    return out


class _Tree:
    """Octree of one system, level by level, of particles in key order.  Centres for the opening
    decisions in the tree precision (sums in octant order, each addition rounded; in double for
    the mixed tree, rounded once); centres and moment sums of the pseudo-particles in double."""

    def __init__(self, pos, u, leaf_max, precision):
        key, self.mn, self.side = _morton(pos)
        self.order = torch.argsort(key, stable=True)
        self.x, self.xd = pos[self.order], pos[self.order].double()
        self.ud = u[self.order].double()
        key = key[self.order]
        n = key.shape[0]
        acc = self.xd if precision == "mixed" else self.x
        d = pos.device
        cm = torch.cat([torch.zeros((1, 9), dtype=torch.float64, device=d),
                        (self.xd[:, :, None] * self.ud[:, None, :]).reshape(n, 9).cumsum(0)])
        live = torch.ones(n, dtype=torch.bool, device=d)   # particles inside an internal cell
        self.lv = []
        for level in range(22):
            pre = key >> (3 * (21 - level))
            idx = torch.nonzero(live).flatten()
            if idx.numel() == 0:
                break
            pl = pre[idx]
            new = torch.ones_like(pl, dtype=torch.bool)
            new[1:] = pl[1:] != pl[:-1]
            start = idx[new]
            cnt = torch.diff(torch.cat([torch.nonzero(new).flatten(),
                                        torch.tensor([idx.numel()], device=d)]))
            leaf = (cnt <= leaf_max) | (level == 21)
            sl = torch.ldexp(self.side, torch.tensor(float(-level), device=d).to(self.side.dtype))
            p = pre[start]
            q = torch.stack([_compact(p >> 2), _compact(p >> 1), _compact(p)], 1).to(pos.dtype)
            end = start + cnt
            self.lv.append(dict(start=start, cnt=cnt, leaf=leaf, lo=self.mn + q * sl, sl=sl,
                                m9=(cm[end] - cm[start]).reshape(-1, 3, 3), key=p))
            live = torch.zeros(n, dtype=torch.bool, device=d)
            keep = torch.repeat_interleave(~leaf, cnt)
            live[idx[keep]] = True
        for level in range(len(self.lv) - 1, -1, -1):
            c = self.lv[level]
            inner = torch.nonzero(~c["leaf"]).flatten()
            c["child0"] = torch.zeros_like(c["start"])
            c["nchild"] = torch.zeros_like(c["start"])
            if inner.numel():
                par = self.lv[level + 1]["key"] >> 3
                new = torch.ones_like(par, dtype=torch.bool)
                new[1:] = par[1:] != par[:-1]
                c0 = torch.nonzero(new).flatten()
                nch = torch.diff(torch.cat([c0, torch.tensor([par.numel()], device=d)]))
                c["child0"][inner], c["nchild"][inner] = c0, nch
            c["sum"] = self._sums(level, acc, "sum", inner)
            c["cd"] = self._sums(level, self.xd, "sx", inner) / c["cnt"][:, None]
            c["w"] = self._sums(level, self.ud, "w", inner)
            c["cen"] = (c["sum"] / c["cnt"][:, None].to(acc.dtype)).to(pos.dtype)
            m9 = c["m9"] - c["cd"][:, :, None] * c["w"][:, None, :]
            m9[c["cnt"] == 1] = 0.0
            c["s"] = 0.5 * (m9 + m9.transpose(1, 2))

    def _sums(self, level, v, name, inner):
        """Cell sums of v: a leaf's particles, then the children, in order."""
        c = self.lv[level]
        sm = v[c["start"]].clone()
        lf = torch.nonzero(c["leaf"] & (c["cnt"] > 1)).flatten()
        for j in range(1, int(c["cnt"][lf].max()) if lf.numel() else 1):
            r = lf[c["cnt"][lf] > j]
            sm[r] = sm[r] + v[c["start"][r] + j]
        if inner.numel():
            ch, c0, nch = self.lv[level + 1], c["child0"][inner], c["nchild"][inner]
            t = ch[name][c0].clone()
            for k in range(1, 8):
                r = nch > k
                t[r] = t[r] + ch[name][c0[r] + k]
            sm[inner] = t
        c[name] = sm
        return sm


def _pair(r, uk, w):
    """T(r) w and the force grad(u_k . T w): (h, f), separations r = target - source."""
    r2 = (r * r).sum(1)
    ir = r2.rsqrt()
    ir3, ir5, ir7 = ir ** 3, ir ** 5, ir ** 7
    bj, bk, a = (w * r).sum(1), (uk * r).sum(1), (w * uk).sum(1)
    h = r * (3 * bj * ir5)[:, None] - w * ir3[:, None]
    f = (r * (3 * a * ir5 - 15 * bk * bj * ir7)[:, None] + uk * (3 * bj * ir5)[:, None]
         + w * (3 * bk * ir5)[:, None])
    return h, f


def _quad(r, uk, s):
    r2 = (r * r).sum(1)
    ir = r2.rsqrt()
    ir5, ir7, ir9 = ir ** 5, ir ** 7, ir ** 9
    m = s[:, 0, 0] + s[:, 1, 1] + s[:, 2, 2]
    sr = (s * r[:, None, :]).sum(2)
    su = (s * uk[:, None, :]).sum(2)
    q, ru, sru = (r * sr).sum(1), (r * uk).sum(1), (sr * uk).sum(1)
    cmq = (3 * m * ir5 - 15 * q * ir7)[:, None]
    cr = (105 * q * ru * ir9 - 30 * sru * ir7 - 15 * m * ru * ir7)[:, None]
    h = -(6 * ir5[:, None] * sr + cmq * r)
    f = -(6 * ir5[:, None] * su - (30 * ru * ir7)[:, None] * sr + cr * r + cmq * uk)
    return h, f


def _lj(r):
    r2 = (r * r).sum(1)
    s6 = (1.0 / r2) ** 3
    return r * (24.0 * (s6 * s6 - s6) / r2)[:, None]


def _bh(pos, u, theta, leaf_max, precision, ds, lj=True, quad=False, grad=False):
    """Barnes-Hut field and force (with the LJ force) in 64 bits, in the given order; with grad
    also the reverse sums over the cells and particles that served as sources."""
    t = _Tree(pos, u, leaf_max, precision)
    n, d, rt = pos.shape[0], pos.device, pos.dtype
    th2 = torch.tensor(theta * theta, dtype=torch.float64).to(rt).item()
    rc2 = torch.tensor(LJ_RCUT * LJ_RCUT, dtype=torch.float64).to(rt).item()
    H = torch.zeros((n, 3), dtype=torch.float64, device=d)
    F, S = torch.zeros_like(H), torch.zeros_like(H)
    G, Q = torch.zeros_like(H), torch.zeros_like(H)
    cellG = [torch.zeros_like(c["cd"]) for c in t.lv] if grad else None
    cellQ = [torch.zeros_like(c["cd"]) for c in t.lv] if grad else None
    step = 1 << 16

    def add(p, xs, w, mark, cells=None, level=0, srcs=None, sym=None):
        for a in range(0, p.numel(), 1 << 24):
            pp = p[a:a + (1 << 24)]
            r = t.xd[pp] - xs[a:a + (1 << 24)]
            ok = (r * r).sum(1) > 0
            if not bool(ok.all()):
                r = torch.where(ok[:, None], r, torch.full_like(r, 1e18))
            ww = w[a:a + (1 << 24)]
            h, f = _pair(r, t.ud[pp], ww)
            if grad:
                gg, _ = _pair(r, ww, t.ud[pp])
                if cells is not None:
                    cc = cells[a:a + (1 << 24)]
                    cellG[level].index_add_(0, cc, gg)
                    cellQ[level].index_add_(0, cc, f / t.lv[level]["cnt"][cc][:, None])
                else:
                    G.index_add_(0, srcs[a:a + (1 << 24)], gg)
                    Q.index_add_(0, srcs[a:a + (1 << 24)], f)
            if sym is not None:
                h2, f2 = _quad(r, t.ud[pp], sym[a:a + (1 << 24)])
                h, f = h + h2, f + f2
            H.index_add_(0, pp, h)
            F.index_add_(0, pp, f)
            if mark and lj:
                x = t.x[pp] - t.x[srcs[a:a + (1 << 24)]]
                r2 = (x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1]) + x[:, 2] * x[:, 2]
                near = (r2 < rc2) & (r2 > 0)
                S.index_add_(0, pp[near], _lj(r[near]))

    for b in range(0, n, step):
        p = torch.arange(b, min(n, b + step), device=d)
        c = torch.zeros_like(p)
        for level, L in enumerate(t.lv):
            if p.numel() == 0:
                break
            x, cen = t.x[p], L["cen"][c]
            dx = x - cen
            d2 = (dx[:, 0] * dx[:, 0] + dx[:, 1] * dx[:, 1]) + dx[:, 2] * dx[:, 2]
            acc = (L["sl"] * L["sl"]) < d2 * th2
            lo = L["lo"][c]
            below, above = lo - x, x - (lo + L["sl"])
            gap = torch.maximum(above, torch.clamp(below, min=0))
            b2 = (gap[:, 0] * gap[:, 0] + gap[:, 1] * gap[:, 1]) + gap[:, 2] * gap[:, 2]
            inside = (p >= L["start"][c]) & (p < L["start"][c] + L["cnt"][c])
            acc &= ~(b2 < rc2) & ~inside
            a = torch.nonzero(acc).flatten()
            add(p[a], L["cd"][c[a]], L["w"][c[a]], False, c[a], level,
                sym=L["s"][c[a]] if quad else None)
            lf = torch.nonzero(~acc & L["leaf"][c]).flatten()
            if lf.numel():
                pl, cl = p[lf], c[lf]
                for j in range(int(L["cnt"][cl].max())):
                    src = L["start"][cl] + j
                    r = (L["cnt"][cl] > j) & (src != pl)
                    add(pl[r], t.xd[src[r]], t.ud[src[r]], True, srcs=src[r])
            o = torch.nonzero(~acc & ~L["leaf"][c]).flatten()
            k = L["nchild"][c[o]]
            first = torch.repeat_interleave(L["child0"][c[o]] - (k.cumsum(0) - k), k)
            p = torch.repeat_interleave(p[o], k)
            c = first + torch.arange(p.numel(), device=d)
    back = torch.empty_like(t.order)
    back[t.order] = torch.arange(n, device=d)
    if grad:
        for L, g, q in zip(t.lv, cellG, cellQ):
            sel = torch.repeat_interleave(torch.arange(L["cnt"].numel(), device=d), L["cnt"])
            off = torch.arange(sel.numel(), device=d) - (L["cnt"].cumsum(0) - L["cnt"])[sel]
            part = L["start"][sel] + off
            G[part] += g[sel]
            Q[part] += q[sel]
        gu, gp = -0.5 * ds * (H + G), -0.5 * ds * (F - Q)
        e = float(-0.5 * ds * (t.ud * H).sum())
        return e, gp[back], gu[back]
    return (ds * H)[back], (ds * F + S)[back]


def _philox(step, n):
    """Six normals per particle (Philox4x32-10 keyed by the seed 7, Box-Muller)."""
    M = 0xFFFFFFFF

    def mul(a, b):
        lo, hi = (a & 0xFFFF) * b, (a >> 16) * b
        full_lo = (lo + ((hi & 0xFFFF) << 16))
        return (hi >> 16) + (full_lo >> 32), full_lo & M

    ids = torch.arange(n, device=_dev(), dtype=torch.int64)
    words = []
    for block in (0, 1):
        c = [torch.full_like(ids, step), torch.zeros_like(ids), ids, torch.full_like(ids, block)]
        k0, k1 = 7, 0
        for r in range(10):
            if r:
                k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
            h0, l0 = mul(c[0], 0xD2511F53)
            h1, l1 = mul(c[2], 0xCD9E8D57)
            c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        words += c
    z = []
    for a, b in ((0, 1), (2, 3), (4, 5)):
        rad = torch.sqrt(-2.0 * torch.log((words[a].double() + 1.0) * 2.0 ** -32))
        ang = words[b].double() * (2.0 * math.pi * 2.0 ** -32)
        z += [rad * torch.cos(ang), rad * torch.sin(ang)]
    return torch.stack(z[:3], 1), torch.stack(z[3:], 1)


def _wall(w):
    wc = w.clamp(min=0.01)
    s6 = (0.5 / wc) ** 6
    return torch.where(w < 0.5, 24.0 * (s6 * s6 - s6) / wc, torch.zeros_like(w))


def _step(x, u, v, w, h, f, hext, hi, gamma, xi_t, xi_r):
    f = f + _wall(x + 0.5) - _wall(hi + 0.5 - x)
    torque = torch.linalg.cross(u, h + hext)
    xn = x + DT * v
    vn = v + DT * (f - gamma * v) + math.sqrt(2.0 * gamma * KT * DT) * xi_t
    wn = (w + DT * (torque - gamma * w) / INERTIA
          + math.sqrt(2.0 * gamma * KT * DT) / INERTIA * xi_r)
    un = u + DT * torch.linalg.cross(w, u)
    return xn, un / un.norm(dim=1, keepdim=True), vn, wn


def exact(case, seed):
    kind = case["kind"]
    if kind == "sensitivity":
        return None  # reverse mode through several steps: no short 64-bit restatement
    s = _inputs(case, seed)
    pos, u = s["pos"], s["u"]
    if kind == "order":
        key, _, _ = _morton(pos)
        order = torch.argsort(key, stable=True)
        return dict(keys=key[order], order=order.to(torch.int32))
    if kind == "allpairs":
        x, m = pos.double(), u.double()
        n = x.shape[0]
        H, F = torch.zeros_like(x), torch.zeros_like(x)
        rows = max(1, (1 << 23) // n)
        rc2 = torch.tensor(LJ_RCUT * LJ_RCUT, dtype=pos.dtype).item()
        for a in range(0, n, rows):
            k = min(n, a + rows) - a
            r = (x[a:a + k, None, :] - x[None, :, :]).reshape(-1, 3)
            d3 = pos[a:a + k, None, :] - pos[None, :, :]
            r2 = (d3[..., 0] * d3[..., 0] + d3[..., 1] * d3[..., 1]) + d3[..., 2] * d3[..., 2]
            zero = (r * r).sum(1) == 0
            r = torch.where(zero[:, None], torch.full_like(r, 1e18), r)
            uk = m[a:a + k, None, :].expand(k, n, 3).reshape(-1, 3)
            h, f = _pair(r, uk, m[None].expand(k, n, 3).reshape(-1, 3))
            near = ((r2 < rc2) & (r2 > 0)).reshape(-1)
            f[near] += _lj(r[near])
            H[a:a + k], F[a:a + k] = h.reshape(k, n, 3).sum(1), f.reshape(k, n, 3).sum(1)
        return dict(h=H, f=F)
    theta, leaf, prec = case["theta"], case["leaf_max"], case["precision"]
    if kind == "field":
        h, f = _bh(pos, u, theta, leaf, prec, 1.0, quad=bool(case["quad"]))
        return dict(h=h, f=f)
    if kind == "grad":
        e, gp, gu = _bh(pos, u, theta, leaf, prec, 1.0, lj=False, grad=True)
        return dict(energy=e, grad_pos=gp, grad_u=gu)
    # time steps
    x, m, v, w = (s[k].double() for k in ("pos", "u", "vel", "omega"))
    n = x.shape[0]
    if kind == "batch":
        own = torch.repeat_interleave(torch.arange(len(s["sizes"])),
                                      torch.tensor(s["sizes"])).to(x.device)
        hext = torch.tensor(s["fields"], device=x.device)[own]
        hi = torch.tensor(s["sides"], device=x.device)[own][:, None]
        cuts = np.concatenate([[0], np.cumsum(s["sizes"])])
        mom = torch.zeros((len(s["sizes"]), 4), dtype=torch.float64, device=x.device)
    else:
        hext = torch.tensor(s["h_ext"], dtype=torch.float64, device=x.device)
        hi, cuts, mom = s["side"], [0, n], None
    for k in range(case["steps"]):
        xr, ur = x.to(pos.dtype), m.to(pos.dtype)
        parts = [_bh(xr[a:b], ur[a:b], theta, leaf, prec, s["dip_scale"])
                 for a, b in zip(cuts[:-1], cuts[1:])]
        h, f = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
        if mom is not None:
            mom.index_add_(0, own, torch.cat([m, h[:, 2:3]], 1))
        xi_t, xi_r = _philox(k, n)
        x, m, v, w = _step(x, m, v, w, h, f, hext, hi, s["gamma"], xi_t, xi_r)
    out = dict(pos=x, u=m, vel=v, omega=w)
    return out if mom is None else dict(moments=mom.cpu().numpy(), **out)
