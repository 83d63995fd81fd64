"""The work a user of the framework has it do, as measurable cases: particle-mesh and P3M force
evaluations, kick-drift-kick steps, graph-replayed runs, ensembles, reverse-mode derivatives and the
power spectrum, from a few thousand particles to 512^3, in both precision modes.

Particle sets are drawn from the seed on the GPU with torch (Zel'dovich displacements of a lattice
with the power-law spectrum of the repository's configurations, the same with Plummer halos on top,
or a random subset of such a lattice for particle numbers that are no cube).  Length unit: the mean
particle spacing is 1.5625 (200/128) unless a case sets the box.

The mixed mode computes forces in FP32 although the API's arrays are FP64; its results are handed
back as FP32 values, the FP64 mode's as FP64 values.

exact() evaluates the same quantities with plain torch in 64 bits: CIC and FFTs on the mesh, all
pairs within the cutoff from a cell list, closed-form split factors, and the transposed derivative
through autograd (mesh) and the pair Jacobian.
"""

import math

import numpy as np
import torch

from paper_1510_07621_gb300 import P3M, Ensemble
from paper_1510_07621_gb300.adjoint import DensityLossRun

SPACING = 200.0 / 128.0
R_S, CUTOFF, SOFT = 1.25, 4.5, 0.02  # mesh cells, split scales, mean spacings


def _case(name, kind, n_p, mesh, **more):
    c = dict(name=name, kind=kind, n_p=n_p, n=n_p ** 3, mesh=mesh, box=n_p * SPACING,
             dist="zeldovich", precision="mixed", short_range=True, omega_m=1.0, omega_lambda=0.0,
             a=0.5, steps=1, step=0.02, graph=False, host=False, sims="")
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: a few thousand particles, no cube, forces once; all latency
        _case("forces_ragged_5003", "forces", 18, 32, n=5003, a=1.0),
        # the all-FP64 comparison configuration: 32^3, one step
        _case("step_fp64_32", "step", 32, 32, box=64.0, precision="fp64", a=0.02, step=0.17),
        # a small box of an ensemble advanced alone, whole steps replayed from CUDA graphs
        _case("steps_graph_48", "step", 48, 48, steps=8, graph=True, a=0.1, step=0.1),
        # FP64 forces on a clustered set (uneven cells, dense halos)
        _case("step_fp64_clustered_48", "step", 48, 48, precision="fp64", dist="clustered",
              a=1.0, step=1e-3),
        # the headline workload: one step of a strongly clustered 128^3 snapshot
        _case("step_clustered_128", "step", 128, 128, dist="clustered", a=1.0, step=1e-3),
        # page-locked host arrays in and out, pure particle-mesh in FP64
        _case("host_pm_fp64_128", "step", 128, 128, precision="fp64", short_range=False,
              host=True, a=0.5, step=0.05),
        # the largest: 134 M particles on a 512^3 mesh, near-uniform
        _case("forces_zeldovich_512", "forces", 512, 512, box=1000.0, a=0.5),
        # mesh-only forces (the 'PM' kick algorithm): sort, deposit, FFTs, gather
        _case("pm_forces_256", "forces", 256, 256, short_range=False, a=0.5),
        # the backward direction: transposed force Jacobian at 128^3
        _case("force_vjp_128", "vjp", 128, 128, a=0.5),
        # one training step: density loss after 4 steps and its gradient (checkpointed sweep)
        _case("gradient_64", "gradient", 64, 64, a=0.05, steps=4, step=0.16),
        # unevenly sized simulations advanced together, one graph launch per step
        _case("ensemble_9", "ensemble", 48, 48, sims="48,48,48,64,64,64,96,96,96", box=100.0,
              steps=2, a=0.05, step=0.16),
        # analysis: power spectrum and sigma_R on a mesh finer than the particle lattice
        _case("spectrum_256", "spectrum", 128, 256, a=1.0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forces", "forces", "step", "step", "vjp", "gradient", "ensemble", "spectrum"])
    dist = rng.choice(["zeldovich", "zeldovich", "clustered"])
    n_p = {"forces": lambda: log(12, 200), "step": lambda: log(12, 128), "vjp": lambda: log(16, 112),
           "gradient": lambda: log(16, 64), "ensemble": lambda: 48,
           "spectrum": lambda: log(16, 192)}[kind]()
    c = _case("", kind, n_p, 0, dist=dist, box=n_p * rng.uniform(0.5, 2.5))
    del c["name"]
    # mesh cells per mean spacing: the mesh is even and leaves at least 3 chaining cells
    c["mesh"] = max(20, 2 * int(round(0.5 * n_p * rng.choice([1.0, 1.0, 1.25, 1.5, 2.0]))))
    c["n"] = n_p ** 3 - (rng.randrange(0, 3 * n_p) if kind in ("forces", "step", "vjp") else 0)
    c["a"] = round(math.exp(rng.uniform(math.log(0.05), 0.0)), 4)
    c["step"] = rng.choice([1e-3, 0.02, 0.1])
    if rng.random() < 0.3 and kind in ("forces", "step"):
        c["omega_m"], c["omega_lambda"] = 0.3, 0.7
    if kind in ("forces", "step"):
        c["short_range"] = rng.random() < 0.75
        if n_p <= 48 or not c["short_range"]:
            c["precision"] = rng.choice(["mixed", "fp64"])
        c["host"] = c["precision"] == "fp64" and rng.random() < 0.5
    if kind == "step":
        c["steps"] = rng.randrange(1, 6)
        c["graph"] = rng.random() < 0.5
    if kind == "gradient":
        c["steps"], c["dist"], c["a"], c["step"] = rng.randrange(2, 7), "zeldovich", 0.05, 0.1
    if kind == "ensemble":
        c["sims"] = ",".join(str(log(20, 96)) for _ in range(rng.randrange(2, 13)))
        c["steps"], c["box"], c["dist"], c["a"] = rng.randrange(1, 4), 100.0, "zeldovich", 0.05
    return c


# ---------------------------------------------------------------- particle sets


def _zeldovich(n_p, box, gen, rms_cells):
    """(3, n_p^3) lattice positions and the displacement field psi, P(k) ~ k^-2 exp(-(k/k_c)^2),
    k_c = k_Nyquist/2, rms |psi| = rms_cells spacings."""
    dev = torch.device("cuda")
    real = torch.float32 if n_p > 256 else torch.float64
    dk = torch.fft.rfftn(torch.randn((n_p,) * 3, generator=gen, device=dev, dtype=real))
    k1 = torch.fft.fftfreq(n_p, 1.0 / n_p, device=dev, dtype=real)
    kz = torch.arange(n_p // 2 + 1, device=dev, dtype=real)
    k2 = k1[:, None, None] ** 2 + k1[None, :, None] ** 2 + kz[None, None, :] ** 2
    kc = n_p / 4.0
    k2[0, 0, 0] = 1.0
    dk *= torch.exp(-0.5 * k2 / kc ** 2) * k2.rsqrt() / k2
    dk[0, 0, 0] = 0.0
    del k2
    psi = torch.empty((3, n_p ** 3), dtype=torch.float64, device=dev)
    for d, kd in enumerate((k1[:, None, None], k1[None, :, None], kz[None, None, :])):
        kd = torch.where(kd.abs() * 2 == n_p, torch.zeros_like(kd), kd)
        psi[d] = torch.fft.irfftn(1j * kd * dk, s=(n_p,) * 3).reshape(-1)
    psi *= rms_cells * (box / n_p) / psi.square().sum(0).mean().sqrt()
    q1 = torch.arange(n_p, device=dev, dtype=torch.float64) * (box / n_p)
    pos = torch.stack([q.reshape(-1) for q in torch.meshgrid(q1, q1, q1, indexing="ij")])
    return pos, psi


def _particles(n_p, n, box, dist, a, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    pos, psi = _zeldovich(n_p, box, gen, 2.0 if dist == "clustered" else 0.2)
    pos += psi
    mom = psi.mul_(math.sqrt(a))
    if dist == "clustered":  # 35 % of the particles in Plummer spheres, dN/d(occupancy) ~ occ^-2
        total = n_p ** 3
        n_move = int(0.35 * total)
        n_h = max(1, n_move // 400)
        u = torch.rand(n_h, generator=gen, device=dev, dtype=torch.float64)
        w = 1.0 / u.clamp_min(1e-3)
        occ = torch.floor(w / w.sum() * n_move).long()
        occ[0] += n_move - occ.sum()
        centres = pos[:, torch.randint(total, (n_h,), generator=gen, device=dev)]
        who = torch.randperm(total, generator=gen, device=dev)[:n_move]
        owner = torch.repeat_interleave(torch.arange(n_h, device=dev), occ)
        rs = 0.15 * (box / n_p) * (occ.clamp_min(1) / 100.0) ** (1.0 / 3.0)
        v = torch.rand((3, n_move), generator=gen, device=dev, dtype=torch.float64)
        r = rs[owner] / torch.sqrt(v[0].clamp(1e-6, 0.999) ** (-2.0 / 3.0) - 1.0)
        r = torch.minimum(r, 10.0 * rs[owner])
        ct = 2.0 * v[1] - 1.0
        st, ph = torch.sqrt((1.0 - ct * ct).clamp_min(0.0)), 2.0 * math.pi * v[2]
        pos[:, who] = centres[:, owner] + torch.stack([r * st * torch.cos(ph), r * st * torch.sin(ph), r * ct])
    pos = torch.remainder(pos, box)
    pos[pos >= box] = 0.0
    if n < n_p ** 3:
        keep = torch.randperm(n_p ** 3, generator=gen, device=dev)[:n]
        pos, mom = pos[:, keep].contiguous(), mom[:, keep].contiguous()
    return pos, mom


def _schedule(c):
    return [c["a"] * (1.0 + c["step"]) ** k for k in range(c["steps"] + 1)]


def _sim(c, n, mesh, box, stream=None):
    return P3M(box, n, mesh, R_S, CUTOFF, c["omega_m"], c["omega_lambda"], precision=c["precision"],
               softening=SOFT, short_range=c["short_range"], stream=stream)


def _sims(c, seed):
    """(n_p, n, mesh, box, seed) of each simulation of the case."""
    if c["kind"] != "ensemble":
        return [(c["n_p"], c["n"], c["mesh"], c["box"], seed)]
    sizes = [int(v) for v in c["sims"].split(",")]
    return [(p, p ** 3, max(20, p + p % 2), c["box"], 1000 * seed + k) for k, p in enumerate(sizes)]


def _field(shape, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 77)
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _gradient_inputs(c, seed):
    """Lattice, displacement field and target density contrast of a training step."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    q, psi = _zeldovich(c["n_p"], c["box"], gen, 0.2)
    # a lattice offset keeps undisplaced particles off the mesh planes
    q += 0.37 * c["box"] / c["mesh"]
    return q, psi, 0.5 * _field((c["mesh"] ** 3,), seed)


# ---------------------------------------------------------------- the cases


def prepare(case, seed):
    c = case
    s = {"c": c, "a": _schedule(c)}
    if c["kind"] == "gradient":
        s["sim"] = _sim(c, c["n"], c["mesh"], c["box"])
        s["q"], psi, s["target"] = _gradient_inputs(c, seed)
        s["psi"] = psi.requires_grad_(True)
        return s
    parts = _sims(c, seed)
    # graph replay needs streams of the program's own
    own = c["kind"] == "ensemble" or (c["graph"] and c["kind"] == "step")
    s["streams"] = [torch.cuda.Stream() for _ in parts] if own else []
    s["sims"], s["in"], s["out"] = [], [], []
    for k, (n_p, n, mesh, box, sd) in enumerate(parts):
        s["sims"].append(_sim(c, n, mesh, box, s["streams"][k] if own else None))
        pm = _particles(n_p, n, box, c["dist"], c["a"], sd)
        out = [torch.empty((3, n), dtype=torch.float64, device="cuda")
               for _ in range({"forces": 1, "vjp": 1, "spectrum": 0}.get(c["kind"], 3))]
        if c["host"]:
            pm = [x.cpu().pin_memory() for x in pm]
            out = [x.cpu().pin_memory() for x in out]
        s["in"].append(pm)
        s["out"].append(out)
    if c["kind"] == "vjp":
        s["v"] = _field((3, c["n"]), seed)
    if c["kind"] == "ensemble":
        s["ens"] = Ensemble(s["sims"], own_streams=False)
    torch.cuda.synchronize()
    return s


def _give(c, tensors):
    return [t if c["precision"] == "fp64" else t.float() for t in tensors]


def run(state):
    s, c, a = state, state["c"], state["a"]
    if c["kind"] == "gradient":
        psi = s["psi"]
        psi.grad = None
        loss = DensityLossRun.apply(psi, s["sim"], s["q"], a, s["target"], 2)
        loss.backward()
        return _give(c, [loss.detach(), psi.grad])
    main = torch.cuda.current_stream()
    for st in s["streams"]:
        st.wait_stream(main)
    for sim, (pos, mom) in zip(s["sims"], s["in"]):
        sim.set_particles(pos, mom, a=a[0])
    sim, out = s["sims"][0], s["out"][0]
    if c["kind"] == "forces":
        sim.forces(a[0], out=out[0])
        return _give(c, out)
    if c["kind"] == "vjp":
        sim.force_vjp(s["v"], out[0])
        return _give(c, out)
    if c["kind"] == "spectrum":
        k, p, modes, sigma = sim.power_spectrum(tophat_radius=8.0)
        return [k, p, modes, sigma]
    if c["kind"] == "ensemble":
        s["ens"].run(a)
        for m, o in zip(s["sims"], s["out"]):
            m.get_particles(*o)
        for st in s["streams"]:
            main.wait_stream(st)
        return [x for o in s["out"] for x in _give(c, o)]
    if c["graph"]:
        sim.run_steps(a)
    else:
        for k in range(len(a) - 1):
            sim.step(a[k], a[k + 1] - a[k])
    sim.get_particles(*out)
    for st in s["streams"]:
        main.wait_stream(st)
    return _give(c, out)


def work(case):
    """What one pass cannot do without: particle state read and written once per evaluation, the
    mesh through its transforms, and the pair arithmetic of the accepted pairs."""
    c = case
    real = 8 if c["precision"] == "fp64" else 4
    out = {"bytes": 0.0, "flops": 0.0}
    evals = {"forces": 1, "vjp": 1, "spectrum": 1}.get(c["kind"], c["steps"] + 1)
    if c["kind"] == "gradient":  # forward, recomputed forward, and one transposed force per state
        evals = 3 * (c["steps"] + 1)
    for n_p, n, mesh, box, _ in _sims(c, 0):
        m3 = float(mesh) ** 3
        per = 48.0 * n if c["kind"] in ("forces", "vjp") else 24.0 * n if c["kind"] == "spectrum" else 72.0 * n
        meshes = 2 if c["kind"] == "spectrum" else 8  # counts, spectrum, three forces each way
        out["bytes"] += evals * (per + meshes * real * m3)
        fft = 2.5 * m3 * math.log2(m3)
        out["flops"] += evals * fft * (1 if c["kind"] == "spectrum" else 4)
        if c["short_range"] and c["kind"] != "spectrum":
            rc = R_S * CUTOFF * box / mesh
            near = 4.0 / 3.0 * math.pi * rc ** 3 * n / box ** 3
            if c["dist"] == "clustered":
                near *= 6.0  # measured pairs of the clustered sets over the uniform count
            out["flops"] += evals * near * n * (63 if real == 8 else 39)
    return out


# ---------------------------------------------------------------- 64-bit values in plain torch


class _Exact:
    def __init__(self, c, n, mesh, box):
        self.c, self.n, self.M, self.L = c, n, mesh, box
        self.h = box / mesh
        self.rs = R_S * self.h
        self.rc = CUTOFF * self.rs
        self.eps = SOFT * box / n ** (1.0 / 3.0)
        self.gm = 3.0 * c["omega_m"] * box ** 3 / (8.0 * math.pi * n)
        dev = torch.device("cuda")
        k = 2.0 * math.pi / box * torch.fft.fftfreq(mesh, 1.0 / mesh, device=dev, dtype=torch.float64)
        kz = 2.0 * math.pi / box * torch.arange(mesh // 2 + 1, device=dev, dtype=torch.float64)
        ks = [k[:, None, None], k[None, :, None], kz[None, None, :]]
        k2 = sum(v * v for v in ks)
        k2[0, 0, 0] = 1.0
        g = -4.0 * math.pi * self.gm / self.h ** 3 / k2
        if c["short_range"]:
            g = g * torch.exp(-k2 * self.rs ** 2)
        for v in ks:
            g = g / torch.sinc(v * (0.5 * self.h / math.pi)) ** 4
        g[0, 0, 0] = 0.0
        self.green = g
        nyq = math.pi * mesh / box
        self.kg = [torch.where((v.abs() - nyq).abs() < 1e-9 * nyq, torch.zeros_like(v), v) for v in ks]

    def stencil(self, x):
        u = x / self.h
        i0 = torch.floor(u.detach())
        f = u - i0
        i0 = i0.long()
        for a in range(2):
            for b in range(2):
                for e in range(2):
                    w = ((f[0] if a else 1 - f[0]) * (f[1] if b else 1 - f[1]) * (f[2] if e else 1 - f[2]))
                    M = self.M
                    yield ((i0[0] + a) % M * M + (i0[1] + b) % M) * M + (i0[2] + e) % M, w

    def counts(self, x):
        rho = torch.zeros(self.M ** 3, dtype=torch.float64, device=x.device)
        for node, w in self.stencil(x):
            rho = rho.index_add(0, node, w)
        return rho

    def mesh_force(self, x):
        M = self.M
        rk = torch.fft.rfftn((self.counts(x) - self.n / M ** 3).reshape(M, M, M)) * self.green
        out = []
        for d in range(3):
            e = torch.fft.irfftn(-1j * self.kg[d] * rk, s=(M, M, M)).reshape(-1)
            out.append(sum(w * e[node] for node, w in self.stencil(x)))
        return torch.stack(out)

    def pairs(self, x):
        """Chunks (i, j, d, r2) of all unordered pairs with 0 < r < r_c, d = x_j - x_i."""
        L, rc, n = self.L, self.rc, self.n
        nc = int(math.floor(L / rc))
        x = x.detach()
        cc = (x * (nc / L)).long().clamp_(max=nc - 1)
        cell = (cc[2] * nc + cc[1]) * nc + cc[0]
        order = torch.argsort(cell)
        xs, cc = x[:, order].contiguous(), cc[:, order]
        start = torch.zeros(nc ** 3 + 1, dtype=torch.long, device=x.device)
        start[1:] = torch.bincount(cell, minlength=nc ** 3).cumsum(0)
        x32 = xs.float()
        far2 = (rc * (1 + 1e-4) + 1e-6 * L) ** 2
        slots = torch.arange(n, device=x.device)
        for k in range(14):  # half of the 27 neighbour cells: pairs are visited once
            off = (k % 3 - 1, k // 3 % 3 - 1, k // 9 - 1)
            nb = [cc[d] + off[d] for d in range(3)]
            img = L * torch.stack([(v >= nc).double() - (v < 0).double() for v in nb])
            w = [v % nc for v in nb]
            q = (w[2] * nc + w[1]) * nc + w[0]
            first, last = start[q], start[q + 1]
            if k == 13:  # the own cell: later slots only
                first = slots + 1
            count = (last - first).clamp_min(0)
            total = count.cumsum(0)
            cuts = torch.searchsorted(total, torch.arange(0, int(total[-1]) + 1, 60_000_000, device=x.device)).tolist()
            cuts = sorted(set([0] + cuts[1:] + [n]))
            for lo, hi in zip(cuts, cuts[1:]):
                cn = count[lo:hi]
                if not int(cn.sum()):
                    continue
                i = torch.repeat_interleave(slots[lo:hi], cn)
                begin = cn.cumsum(0) - cn
                j = torch.arange(i.numel(), device=x.device) + (first[lo:hi] - begin)[i - lo]
                r2 = None
                for d in range(3):
                    t = x32[d, j] - (x32[d] - img[d].float())[i]
                    r2 = t * t if r2 is None else r2.addcmul_(t, t)
                keep = (r2 < far2).nonzero()[:, 0]
                i, j = i[keep], j[keep]
                dd = torch.stack([(xs[d, j] - xs[d, i]) + img[d, i] for d in range(3)])
                r2 = (dd * dd).sum(0)
                ok = ((r2 < rc * rc) & (r2 > 0)).nonzero()[:, 0]
                yield order[i[ok]], order[j[ok]], dd[:, ok], r2[ok]

    def split(self, r2):
        """h = g(r/r_s) (r^2 + eps^2)^-3/2 and r."""
        r = torch.sqrt(r2)
        u = 0.5 * r / self.rs
        g = torch.erfc(u) + (2.0 / math.sqrt(math.pi)) * u * torch.exp(-u * u)
        s = torch.rsqrt(r2 + self.eps ** 2)
        return g * s * s * s, r, g, s

    def forces(self, x):
        acc = self.mesh_force(x)
        if self.c["short_range"]:
            for i, j, d, r2 in self.pairs(x):
                f = self.gm * self.split(r2)[0] * d
                for e in range(3):
                    acc[e].index_add_(0, i, f[e])
                    acc[e].index_add_(0, j, f[e], alpha=-1)
        return acc

    def vjp(self, x, v):
        """(dA/dx)^T v."""
        y = x.detach().clone().requires_grad_(True)
        with torch.enable_grad():
            (out,) = torch.autograd.grad((self.mesh_force(y) * v).sum(), y)
        out = out.clone()
        if self.c["short_range"]:
            for i, j, d, r2 in self.pairs(x):
                h, r, g, s = self.split(r2)
                gd = -(r2 / self.rs ** 3) * torch.exp(-0.25 * r2 / self.rs ** 2) / (2 * math.sqrt(math.pi))
                hr = gd * s ** 3 / r - 3.0 * g * s ** 5
                w = v[:, j] - v[:, i]
                o = self.gm * (h * w + hr * (d * w).sum(0) * d)
                for e in range(3):
                    out[e].index_add_(0, i, o[e])
                    out[e].index_add_(0, j, o[e], alpha=-1)
        return out

    def factor(self, a1, a2, power):
        """int da / (a^power H(a))."""
        om, ol = self.c["omega_m"], self.c["omega_lambda"]
        x, w = np.polynomial.legendre.leggauss(64)
        a = 0.5 * (a2 - a1) * x + 0.5 * (a2 + a1)
        hub = np.sqrt(om / a ** 3 + (1.0 - om - ol) / a ** 2 + ol)
        return float(0.5 * (a2 - a1) * np.sum(w / (a ** power * hub)))

    def kdk(self, x, p, acc, a1, a2):
        am = 0.5 * (a1 + a2)
        p = p + self.factor(a1, am, 2) * acc
        x = torch.remainder(x + self.factor(a1, a2, 3) * p, self.L)
        acc = self.forces(x)
        return x, p + self.factor(am, a2, 2) * acc, acc


def _exact_gradient(c, seed):
    q, psi, target = _gradient_inputs(c, seed)
    e, a = _Exact(c, c["n"], c["mesh"], c["box"]), _schedule(c)
    x, p = torch.remainder(q + psi, c["box"]), math.sqrt(a[0]) * psi
    acc, states = e.forces(x), [x]
    for k in range(len(a) - 1):
        x, p, acc = e.kdk(x, p, acc, a[k], a[k + 1])
        states.append(x)
    y = x.detach().clone().requires_grad_(True)
    with torch.enable_grad():
        loss = (e.counts(y) * (c["mesh"] ** 3 / c["n"]) - 1.0 - target).square().sum()
        (lx,) = torch.autograd.grad(loss, y)
    lp = torch.zeros_like(lx)
    mid = [0.5 * (u + v) for u, v in zip(a, a[1:])]
    for k in range(len(a) - 2, -1, -1):
        kick = e.factor(mid[k], a[k + 1], 2)
        if k + 1 < len(mid):
            kick += e.factor(a[k + 1], mid[k + 1], 2)
        if k + 2 < len(a):  # (lp = 0 before the last drift)
            lx = lx + kick * e.vjp(states[k + 1], lp)
        lp = lp + e.factor(a[k], a[k + 1], 3) * lx
    lx = lx + e.factor(a[0], mid[0], 2) * e.vjp(states[0], lp)
    return [loss.detach(), lx + math.sqrt(a[0]) * lp]


def _exact_spectrum(c, x):
    M, L, n = c["mesh"], c["box"], c["n"]
    e = _Exact(c, n, M, L)
    dk = torch.fft.rfftn((e.counts(x) - n / M ** 3).reshape(M, M, M)) / n
    i1 = torch.fft.fftfreq(M, 1.0 / M, device=x.device, dtype=torch.float64)
    iz = torch.arange(M // 2 + 1, device=x.device, dtype=torch.float64)
    idx = [i1[:, None, None], i1[None, :, None], iz[None, None, :]]
    nk = torch.sqrt(sum(v * v for v in idx))
    p = dk.abs() ** 2
    for v in idx:
        p = p / torch.sinc(v / M) ** 4
    w = torch.where((iz == 0) | (iz == M // 2), 1.0, 2.0).expand_as(nk).double()
    kr = 2.0 * math.pi / L * nk * 8.0
    kr[0, 0, 0] = 1.0
    win = 3.0 * (torch.sin(kr) - kr * torch.cos(kr)) / kr ** 3
    win = torch.where(kr < 1e-3, 1.0 - kr * kr / 10.0, win)
    p[0, 0, 0] = 0.0
    sigma = (w * p * win * win).sum().sqrt()
    shell = torch.floor(nk + 0.5).long().reshape(-1) - 1
    ok = ((shell >= 0) & (shell < M // 2)).nonzero()[:, 0]
    sums = []
    for v in (w * p, w * nk * (2.0 * math.pi / L), w):
        sums.append(torch.zeros(M // 2, dtype=torch.float64, device=x.device).index_add_(0, shell[ok], v.reshape(-1)[ok]))
    return [(sums[1] / sums[2]).cpu().numpy(), (L ** 3 * sums[0] / sums[2]).cpu().numpy(),
            sums[2].cpu().numpy(), float(sigma)]


def exact(case, seed):
    c = case
    cost = sum(n for _, n, _, _, _ in _sims(c, seed)) * (6.0 if c["dist"] == "clustered" else 1.0)
    evals = {"forces": 1, "vjp": 2}.get(c["kind"], c["steps"] + 1)
    # pairs per particle grow with the cells' occupancy
    near = (R_S * CUTOFF * c["n_p"] / c["mesh"]) ** 3 / 178.0
    if c["short_range"] and c["kind"] != "spectrum" and cost * evals * near > 3.0e7 or c["n"] > 3e7:
        return None
    with torch.no_grad():
        if c["kind"] == "gradient":
            return _exact_gradient(c, seed)
        result = []
        for n_p, n, mesh, box, sd in _sims(c, seed):
            x, p = _particles(n_p, n, box, c["dist"], c["a"], sd)
            if c["kind"] == "spectrum":
                return _exact_spectrum(c, x)
            e, a = _Exact(c, n, mesh, box), _schedule(c)
            if c["kind"] == "vjp":
                result.append(e.vjp(x, _field((3, n), seed)))
                continue
            acc = e.forces(x)
            if c["kind"] == "forces":
                result.append(acc)
                continue
            for k in range(len(a) - 1):
                x, p, acc = e.kdk(x, p, acc, a[k], a[k + 1])
            result += [x, p, acc]
        return result
