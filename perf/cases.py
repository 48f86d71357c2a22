"""The workloads whose time a user of this library pays for, each as one call through the public binding.

listed() are the workloads, draw() gives further ones of the same ranges, prepare() makes what a
program holds before the call (domains, a batch, a network, device fields), run() is one pass,
work() its algorithmic bytes and flops, exact() the same pass in FP64 with plain torch.

Kinds:
  pipe       straight pipe, body-force driven, periodic along z: `steps` time steps, then rho and u of
             the fluid cells into device arrays (a run between two outputs)
  aneurysm   seeded synthetic aneurysm (Bouzidi walls, pulsatile inlet, outlet with its absorbing
             layer): the same; with `monitor` also a running-mean sample, FP64 diagnostics, probes
  batch      several uneven aneurysms advanced together by one batch, then each one's fields
  corrector  a fine snapshot restricted onto the coarse grid and the network's correction for it
  train      training steps of the network on such a pair
  corrected  a coarse run with the network in the loop: a batch chunk, one correction, dense fields
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2101_11107_gb300 import inputs as I
from paper_2101_11107_gb300 import lbm

VALUE_BYTES = {"fp32": 4, "fp16": 2, "bf16": 2}
U_SCALE, RHO_SCALE, DU_SCALE = 0.05, 0.01, 0.005


def listed():
    return [
        # the smallest real run: the 32x32x64 validation pipe, default launch configuration, a few
        # microseconds a step -- launches and latency
        dict(name="poiseuille32_fp32", kind="pipe", nx=32, ny=32, nz=64, radius=12.0, bouzidi=False, drive="steady",
             storage="fp32", scheme="esoteric", collision="chm", steps=20, tune=False),
        # the headline workload, the 64x64x256 Womersley pipe, autotuned as the benchmark does: in place, ...
        dict(name="womersley_fp32", kind="pipe", nx=64, ny=64, nz=256, radius=28.0, bouzidi=False, drive="pulse",
             storage="fp32", scheme="esoteric", collision="chm", steps=20, tune=True),
        # ... with two population arrays (the scheme of the slab decomposition), ...
        dict(name="womersley_fp32_ab", kind="pipe", nx=64, ny=64, nz=256, radius=28.0, bouzidi=False, drive="pulse",
             storage="fp32", scheme="ab", collision="chm", steps=20, tune=True),
        # ... and in half the memory
        dict(name="womersley_fp16", kind="pipe", nx=64, ny=64, nz=256, radius=28.0, bouzidi=False, drive="pulse",
             storage="fp16", scheme="esoteric", collision="chm", steps=20, tune=True),
        # a long high-resolution pipe with interpolated walls, odd extents: a state several times L2
        dict(name="pipe_large_fp32", kind="pipe", nx=131, ny=127, nz=252, radius=58.3, bouzidi=True, drive="pulse",
             storage="fp32", scheme="esoteric", collision="chm", steps=20, tune=False),
        # the paper's kind of run: a 256^3 vessel with an aneurysm, every boundary rule in use
        dict(name="aneurysm256_fp32", kind="aneurysm", edge=256, geometry=11, storage="fp32", scheme="esoteric",
             collision="chm", steps=20, tune=True, monitor=False),
        # a monitored run: between outputs, a mean sample, diagnostics and probes; BF16, two arrays
        dict(name="monitored150_bf16_ab", kind="aneurysm", edge=150, geometry=5, storage="bf16", scheme="ab",
             collision="chm", steps=10, tune=False, monitor=True),
        # the operator the paper compares against (stability study), on a small vessel
        dict(name="aneurysm128_trt2", kind="aneurysm", edge=128, geometry=200, storage="fp32", scheme="esoteric",
             collision="trt2", steps=20, tune=False, monitor=False),
        # many patients at once: uneven vessels, FP16, one batch replaying captured steps
        dict(name="batch8_fp16", kind="batch", edges="96,112,144,128,96,160,112,128", storage="fp16", steps=50,
             graph_steps=50, tune=True),
        # evaluation of the learned corrector on a restricted fine snapshot
        dict(name="corrector128", kind="corrector", edge=128, geometry=201),
        # its training
        dict(name="train128", kind="train", edge=128, geometry=202, steps=2, lr=1e-4),
        # the coarse solver with the corrector in the loop every 50 steps
        dict(name="corrected128", kind="corrected", edge=128, geometry=203, steps=50),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["pipe", "pipe", "pipe", "aneurysm", "aneurysm", "aneurysm", "batch", "corrector", "train",
                       "corrected"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    scheme = rng.choice(["esoteric", "esoteric", "ab"])
    collision = rng.choice(["chm", "chm", "chm", "chm", "chm_rates", "srt2", "trt2"])
    tune = rng.random() < 0.5
    if kind == "pipe":
        r = math.exp(rng.uniform(math.log(5.0), math.log(50.0)))
        nx, ny = int(2 * r) + rng.randint(3, 9), int(2 * r) + rng.randint(3, 9)
        return dict(kind=kind, nx=nx, ny=ny, nz=4 * log_int(2, 64), radius=round(r, 2), bouzidi=rng.random() < 0.4,
                    drive=rng.choice(["steady", "pulse"]), storage=storage, scheme=scheme, collision=collision,
                    steps=rng.randint(3, 20), tune=tune)
    if kind == "aneurysm":
        return dict(kind=kind, edge=log_int(48, 200), geometry=rng.randint(1, 400), storage=storage, scheme=scheme,
                    collision=collision, steps=rng.randint(3, 20), tune=tune, monitor=rng.random() < 0.5)
    if kind == "batch":
        edges = [rng.randint(48, 144) for _ in range(rng.randint(2, 8))]
        return dict(kind=kind, edges=",".join(map(str, edges)), storage=storage, steps=rng.randint(20, 50),
                    graph_steps=2 * rng.randint(5, 25), tune=tune)
    edge = 4 * log_int(12, 40)
    if kind == "corrector":
        return dict(kind=kind, edge=edge, geometry=rng.randint(1, 400))
    if kind == "train":
        return dict(kind=kind, edge=edge, geometry=rng.randint(1, 400), steps=rng.randint(1, 2), lr=1e-4)
    return dict(kind=kind, edge=edge, geometry=rng.randint(1, 400), steps=10 * rng.randint(2, 5))


# ------------------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=24)
def _aneurysm(seed, edge):
    return I.aneurysm(seed, edge=edge, period=float(round(15.625 * edge)))


@functools.lru_cache(maxsize=4)
def _pipe(nx, ny, nz, radius, bouzidi, drive):
    if drive == "steady":
        return I.pipe(nx, ny, nz, radius, tau=0.6, g0=(0.0, 0.0, 1e-6 * (12.0 / radius) ** 2), bouzidi=bouzidi)
    nu = 0.05 / 3.0
    return I.pipe(nx, ny, nz, radius, tau=0.55, gamp=(0.0, 0.0, 1e-5 * (28.0 / radius) ** 2),
                  gomega=16.0 * nu / radius ** 2, bouzidi=bouzidi)


def _geometry(case, seed):
    if case["kind"] == "pipe":
        return _pipe(case["nx"], case["ny"], case["nz"], case["radius"], case["bouzidi"], case["drive"])
    g = _aneurysm(case["geometry"], case["edge"])
    return dataclasses.replace(g, wave=I.cardiac_waveform(seed, period=g.wave[2], u_peak=g.wave[3]))


def _members(case, seed):
    out = []
    for k, e in enumerate(int(v) for v in case["edges"].split(",")):
        g = _aneurysm(300 + k, e)
        out.append(dataclasses.replace(g, wave=I.cardiac_waveform(seed + k, period=g.wave[2], u_peak=g.wave[3])))
    return out


def _fields(shape, seed, u_mean=0.0, u_amp=0.004, rho_amp=0.002):
    """A seeded smooth flow field on the box: a mean velocity along z plus a few Fourier modes."""
    rng = np.random.default_rng(seed)
    nz, ny, nx = shape
    ax = [(torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) / n for n in (nx, ny, nz)]
    out = []
    for amp in (u_amp, u_amp, u_amp, rho_amp):
        f = torch.zeros(shape, device="cuda")
        for _ in range(2):
            s = [torch.sin(2 * math.pi * int(rng.integers(1, 4)) * x + float(rng.uniform(0, 6.28))) for x in ax]
            f += amp * float(rng.uniform(0.5, 1.0)) * s[2][:, None, None] * s[1][:, None] * s[0]
        out.append(f)
    out[2] += u_mean * (0.8 + 0.4 * float(rng.random()))
    return 1.0 + out[3], torch.stack(out[:3])


def _initial(g, seed):
    return _fields(g.shape, seed, u_mean=0.02 if g.wave is None else 0.0)


def _rates(case):
    return (1.2, 1.1, 1.05, 0.95) if case.get("collision") == "chm_rates" else (1.0, 1.0, 1.0, 1.0)


def _domain(g, case, seed):
    coll = case.get("collision", "chm")
    dom = lbm.Domain.from_geometry(g, storage=case.get("storage", "fp32"), scheme=case.get("scheme", "esoteric"),
                                   collision="chm" if coll == "chm_rates" else coll, omega_hi=_rates(case))
    dom.init_equilibrium(*_initial(g, seed))
    return dom


def _probes(g, seed, n=32):
    zyx = np.argwhere(g.mask != 0)
    return zyx[np.random.default_rng(seed).integers(0, len(zyx), n)]


def _mask(g):
    return torch.from_numpy((g.mask > 0).astype(np.uint8)).cuda()


def _bulk(m):
    """Fluid cells whose 26 neighbours are all fluid (the cells the correction acts on)."""
    p = torch.nn.functional.pad(1.0 - (m > 0).float(), (1, 1, 1, 1, 1, 1), value=1.0)
    return (torch.nn.functional.max_pool3d(p[None, None], 3, 1)[0, 0] == 0).to(torch.uint8)


def _fine_snapshot(m, seed):
    """A snapshot on the grid twice as fine, solid where the coarse cell is: (rho, u, mask)."""
    fm = m.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2).contiguous()
    rho, u = _fields(fm.shape, seed, u_mean=0.01, u_amp=0.01)
    return rho * fm, u * fm, fm


def _network(g, seed, du_scale=DU_SCALE):
    return lbm.Corrector(g.mask, I.corrector_init_params(seed), U_SCALE, RHO_SCALE, du_scale)


def _compact(dom, out):
    dom.macroscopic_device(out[0], out[1], dense=False)
    return out


def _out(dom):
    n = dom.info()["n_fluid"]
    return torch.empty(n, device="cuda"), torch.empty((3, n), device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("pipe", "aneurysm"):
        g = _geometry(case, seed)
        s = dict(kind=kind, dom=_domain(g, case, seed), steps=case["steps"], monitor=case.get("monitor", False))
        s["out"] = _out(s["dom"])
        if s["monitor"]:
            s["points"] = _probes(g, seed)
            s["dom"].mean_reset()
        if case["tune"]:
            s["dom"].autotune(10)
        return s
    if kind == "batch":
        doms = [_domain(g, case, seed + k) for k, g in enumerate(_members(case, seed))]
        batch = lbm.Batch(doms, graph_steps=case["graph_steps"])
        if case["tune"]:
            batch.autotune(min(10, case["graph_steps"]))
        return dict(kind=kind, doms=doms, batch=batch, outs=[_out(d) for d in doms], steps=case["steps"])
    g = _geometry(case, seed)
    m = _mask(g)
    if kind == "corrected":
        dom = _domain(g, case, seed)
        return dict(kind=kind, dom=dom, batch=lbm.Batch([dom], graph_steps=case["steps"]), mask=m, bulk=_bulk(m),
                    net=_network(g, seed, DU_SCALE / 10), steps=case["steps"])
    if kind == "corrector":
        rho, u, fm = _fine_snapshot(m, seed)
        return dict(kind=kind, net=_network(g, seed), rho=rho, u=u, fine_mask=fm, mask=m, bulk=_bulk(m))
    rho, u, target = _pair(m, seed)
    return dict(kind=kind, net=_network(g, seed), rho=rho, u=u, target=target, mask=m, bulk=_bulk(m),
                steps=case["steps"], lr=case["lr"])


def _pair(m, seed):
    rho, u = _fields(m.shape, seed, u_mean=0.01, u_amp=0.01)
    _, du = _fields(m.shape, seed + 7919, u_amp=0.002)
    return rho * m, u * m, (u + du) * m


# ------------------------------------------------------------------------------ the passes
def run(s):
    kind = s["kind"]
    if kind in ("pipe", "aneurysm"):
        s["dom"].step(s["steps"])
        rho, u = _compact(s["dom"], s["out"])
        if not s["monitor"]:
            return {"rho": rho, "u": u}
        s["dom"].mean_sample()
        diag = s["dom"].diagnostics(raise_unstable=False)
        probes = s["dom"].probe(s["points"])
        rho_mean, u_mean, n = s["dom"].mean(dense=False)
        return {"rho": rho, "u": u, "diag": diag, "probes": probes, "rho_mean": rho_mean, "u_mean": u_mean, "n": n}
    if kind == "batch":
        s["batch"].step(s["steps"])
        return [_compact(d, o) for d, o in zip(s["doms"], s["outs"])]
    if kind == "corrector":
        rho, u = lbm.restrict(s["rho"], s["u"], s["fine_mask"])
        return {"rho": rho, "u": u, "du": s["net"].forward(rho, u, mask=s["mask"], out_mask=s["bulk"])}
    if kind == "train":
        loss = [s["net"].train_step(s["rho"], s["u"], s["target"], s["lr"], mask=s["mask"], out_mask=s["bulk"])
                for _ in range(s["steps"])]
        return {"loss": loss, "params": s["net"].params()}
    s["batch"].step(s["steps"])
    s["net"].apply(s["dom"], mask=s["mask"], out_mask=s["bulk"], gain=0.25)
    rho, u = s["dom"].macroscopic_tensors()
    return {"rho": rho, "u": u}


# ------------------------------------------------------------------------------ algorithmic work
NET_FLOPS = 3 * 27 * 16 * 16 * 2  # per evaluated cell, forward


def _step_work(n, storage, steps):
    return 2.0 * 27 * VALUE_BYTES[storage] * n * steps, 350.0 * n * steps


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = sum(g.nfluid for g in _members(case, 0))
        b, f = _step_work(n, case["storage"], case["steps"])
        return {"bytes": b + 16.0 * n, "flops": f}
    g = _geometry(case, 0)
    n, box = g.nfluid, g.mask.size
    if kind in ("pipe", "aneurysm"):
        b, f = _step_work(n, case["storage"], case["steps"])
        # the export writes 16 B per cell; a monitored run reads the state again and updates FP64 sums
        return {"bytes": b + 16.0 * n + (96.0 * n if case.get("monitor") else 0.0), "flops": f}
    if kind == "corrector":  # fine mask and fields once, coarse fields and du written, layers on fluid cells
        return {"bytes": 8.0 * box + 8 * 16.0 * n + 28.0 * box, "flops": 1.0 * NET_FLOPS * n}
    if kind == "train":      # rho, u, target; activations and their gradients of three layers (32 B per cell)
        return {"bytes": case["steps"] * (28.0 + 6 * 32) * n, "flops": 3.0 * NET_FLOPS * n * case["steps"]}
    b, f = _step_work(n, "fp32", case["steps"])
    return {"bytes": b + 216.0 * n + 16.0 * box, "flops": f + NET_FLOPS * n}


# ------------------------------------------------------------------------------ FP64 reference
_C = [((i % 3) - 1, ((i // 3) % 3) - 1, (i // 9) - 1) for i in range(27)]
_W = [(2 / 3 if c[0] == 0 else 1 / 6) * (2 / 3 if c[1] == 0 else 1 / 6) * (2 / 3 if c[2] == 0 else 1 / 6) for c in _C]


class _Exact:
    """The lattice Boltzmann case in FP64 on a compact cell list: f* of the previous level is the state."""

    def __init__(self, g, case, seed):
        self.g, self.coll, self.om = g, case.get("collision", "chm"), _rates(case)
        dev = "cuda"
        mask = torch.from_numpy(g.mask).to(dev)
        nz, ny, nx = g.shape
        box = torch.nonzero(mask.reshape(-1)).reshape(-1)
        rank = torch.full((mask.numel(),), -1, dtype=torch.int64, device=dev)
        rank[box] = torch.arange(len(box), device=dev)
        self.box, self.n = box, len(box)
        p = [box % nx, (box // nx) % ny, box // (nx * ny)]
        self.kind = mask.reshape(-1)[box]
        self.src = []
        for c in _C:
            ok, q = torch.ones_like(box, dtype=torch.bool), []
            for d, ext in enumerate((nx, ny, nz)):
                v = p[d] - c[d]
                if g.periodic[d]:
                    v = v % ext
                else:
                    ok &= (v >= 0) & (v < ext)
                    v = v.clamp(0, ext - 1)
                q.append(v)
            r = rank[q[0] + nx * (q[1] + ny * q[2])]
            self.src.append(torch.where(ok, r, torch.full_like(r, -1)))
        self.links = None
        if g.links is not None and len(g.links[0]):
            cell = rank[torch.from_numpy(g.links[0]).to(dev)]
            self.links = cell, 26 - torch.from_numpy(g.links[1].astype(np.int64)).to(dev), torch.from_numpy(g.links[2]).to(dev)
        tau = torch.full((self.n,), float(g.tau), dtype=torch.float64, device=dev)
        if g.tau_cell is not None:
            tau = torch.from_numpy(np.ascontiguousarray(g.tau_cell)).to(dev).reshape(-1)[box]
        self.tau = tau
        self.open = []
        ext = (nx, ny, nz)
        for d in range(3):
            for sgn, at in ((1, 0), (-1, ext[d] - 1)):
                sel = torch.nonzero((self.kind >= 2) & (p[d] == at)).reshape(-1) if not g.periodic[d] else box[:0]
                for kind in (2, 3):
                    cells = sel[self.kind[sel] == kind]
                    if len(cells):
                        r2 = sum((p[t][cells].double() + 0.5 - g.inlet_center[t]) ** 2 for t in range(3) if t != d)
                        phi = (2.0 * (1.0 - r2 / g.inlet_radius ** 2)).clamp(min=0.0)
                        self.open.append((cells, d, sgn, kind, phi))
        self.wave = None
        if g.wave is not None:
            a, b, period, peak = g.wave
            t = np.arange(int(period))
            v = a[0] + sum(a[k] * np.cos(2 * np.pi * k * t / period) + b[k - 1] * np.sin(2 * np.pi * k * t / period)
                           for k in range(1, len(a)))
            self.wave = peak * v / v.max()
        self.time = 0
        rho, u = _initial(g, seed)
        rho, u = rho.double().reshape(-1)[box], u.double().reshape(3, -1)[:, box]
        self.post = torch.stack([rho * e for e in self._eq(u)])
        self._stream()

    @staticmethod
    def _eq(u):
        psi = [{0: 2 / 3 - u[d] ** 2, 1: 1 / 6 + (u[d] + u[d] ** 2) / 2, -1: 1 / 6 + (u[d] ** 2 - u[d]) / 2} for d in range(3)]
        return [psi[0][c[0]] * psi[1][c[1]] * psi[2][c[2]] for c in _C]

    def force(self):
        return [self.g.g0[d] + self.g.gamp[d] * math.cos(self.g.gomega * self.time) for d in range(3)]

    def _stream(self):
        post = self.post
        f = torch.empty_like(post)
        for i in range(27):
            s = self.src[i]
            f[i] = torch.where(s >= 0, post[i][s.clamp(min=0)], post[26 - i])
        if self.links is not None:
            cell, al, q = self.links
            flat = torch.stack(self.src)
            far = torch.where(flat[26 - al, cell] >= 0, f[26 - al, cell], f[al, cell])  # f*_b at x + c_a, if fluid
            near, own = f[al, cell], post[al, cell]
            low = torch.where(flat[26 - al, cell] >= 0, 2 * q * near + (1 - 2 * q) * far, near)
            f[al, cell] = torch.where(q < 0.5, low, near / (2 * q) + (2 * q - 1) / (2 * q) * own)
        inflow = float(self.wave[self.time % len(self.wave)]) if self.wave is not None else 0.0
        for cells, d, sgn, kind, phi in self.open:
            h = f[:, cells]
            cn = [sgn * c[d] for c in _C]
            s = sum(h[i] * (1.0 if cn[i] == 0 else 2.0) for i in range(27) if cn[i] <= 0)
            if kind == 2:
                un = inflow * phi
                rho = s / (1.0 - un)
            else:
                rho = torch.ones_like(s)
                un = 1.0 - s / rho
            for i in range(27):
                if cn[i] == 1:
                    h[i] = h[26 - i] + 6.0 * _W[i] * rho * un
            for t in range(3):
                if t != d:
                    mom = sum(c[t] * h[i] for i, c in enumerate(_C) if c[t])
                    for i, c in enumerate(_C):
                        if cn[i] == 1 and c[t]:
                            h[i] = h[i] - c[t] * mom / 6.0
            f[:, cells] = h
        self.f = f

    def fields(self):
        rho = self.f.sum(0)
        gr = self.force()
        u = torch.stack([sum(c[d] * self.f[i] for i, c in enumerate(_C) if c[d]) / rho + 0.5 * gr[d] for d in range(3)])
        return rho, u

    def step(self, n):
        for _ in range(n):
            rho, u = self.fields()
            gr = self.force()
            self.post = self._classical(rho, u, gr) if self.coll in ("srt2", "trt2") else self._moments(rho, u, gr)
            self.time += 1
            self._stream()

    def _moments(self, rho, u, gr):
        """Central Hermite moments: T is a product of 3x3 matrices per axis, rows (1, xi, xi^2 - 1/3)."""
        n, t = self.n, []
        for d in range(3):
            xi = [-1.0 - u[d], -u[d], 1.0 - u[d]]
            t.append(torch.stack([torch.stack([x ** 0 for x in xi]), torch.stack(xi), torch.stack([x * x - 1 / 3 for x in xi])])
                     .permute(2, 0, 1))
        a = self.f.T.reshape(n, 3, 3, 3)  # (z, y, x)
        a = torch.einsum("nij,nzyj->nzyi", t[0], a)
        a = torch.einsum("nij,nzjx->nzix", t[1], a)
        a = torch.einsum("nij,njyx->niyx", t[2], a).reshape(n, 27)
        new = torch.empty_like(a)
        for m in range(27):
            o = m % 3 + (m // 3) % 3 + m // 9
            if o == 0:
                new[:, m] = rho
            elif o == 1:
                new[:, m] = 0.5 * rho * gr[{1: 0, 3: 1, 9: 2}[m]]
            else:
                s = 1.0 / self.tau if o == 2 else self.om[o - 3]
                new[:, m] = (1.0 - s) * a[:, m]
        inv = [torch.linalg.inv(v) for v in t]
        a = torch.einsum("nij,njyx->niyx", inv[2], new.reshape(n, 3, 3, 3))
        a = torch.einsum("nij,nzjx->nzix", inv[1], a)
        a = torch.einsum("nij,nzyj->nzyi", inv[0], a)
        return a.reshape(n, 27).T.contiguous()

    def _classical(self, rho, u, gr):
        """Two relaxation times (one for srt2), second-order equilibrium and force term."""
        wp = 1.0 / self.tau
        wm = wp if self.coll == "srt2" else 1.0 / ((3.0 / 16.0) / (self.tau - 0.5) + 0.5)
        uu = (u * u).sum(0)
        om = torch.empty_like(self.f)
        for i, c in enumerate(_C):
            j = 26 - i
            cu = sum(c[d] * u[d] for d in range(3))
            cf = sum(c[d] * gr[d] for d in range(3)) * rho
            uf = sum(u[d] * gr[d] for d in range(3)) * rho
            even = 0.5 * (self.f[i] + self.f[j]) - _W[i] * rho * (1 + 4.5 * cu ** 2 - 1.5 * uu)
            odd = 0.5 * (self.f[i] - self.f[j]) - _W[i] * rho * 3 * cu
            om[i] = (self.f[i] - wp * even - wm * odd + (1 - wp / 2) * _W[i] * (9 * cu * cf - 3 * uf)
                     + (1 - wm / 2) * _W[i] * 3 * cf)
        return om

    def correct(self, du):
        """du: dense (3, nz, ny, nx); the post-collision state gains f_eq(rho, u + du) - f_eq(rho, u)."""
        rho, u = self.fields()
        d = du.reshape(3, -1)[:, self.box] * (self.kind < 2)
        self.post = self.post + rho * (torch.stack(self._eq(u + d)) - torch.stack(self._eq(u)))
        self._stream()

    def dense(self):
        rho, u = self.fields()
        out = torch.zeros((4, self.g.mask.size), dtype=torch.float64, device="cuda")
        out[0, self.box] = rho
        out[1:, self.box] = u
        return out[0].reshape(self.g.shape), out[1:].reshape(3, *self.g.shape)


def _net64(params, rho, u, m):
    """The three-layer network in FP64: O[0:3] on the dense box."""
    on = (m > 0).double()
    x = torch.zeros((*m.shape, 16), dtype=torch.float64, device="cuda")
    for d in range(3):
        x[..., d] = u[d].double() / U_SCALE * on
    x[..., 3] = (rho.double() - 1.0) / RHO_SCALE * on
    x[..., 4] = on
    nz, ny, nx = m.shape
    for layer in range(3):
        w, b = params[2 * layer], params[2 * layer + 1]
        p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
        y = b
        for o in range(27):
            dx, dy, dz = o % 3, (o // 3) % 3, o // 9
            y = y + p[dz:dz + nz, dy:dy + ny, dx:dx + nx] @ w[o].T
        x = torch.relu(y) if layer < 2 else y
    return x[..., :3].permute(3, 0, 1, 2)


def _params64(seed):
    return [torch.from_numpy(np.asarray(v)).cuda() for v in I.corrector_init_params(seed)]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pipe", "aneurysm"):
        g = _geometry(case, seed)
        e = _Exact(g, case, seed)
        e.step(case["steps"])
        rho, u = e.fields()
        if not case.get("monitor"):
            return {"rho": rho, "u": u}
        flux = [0.0, 0.0]
        for cells, d, sgn, k, _ in e.open:
            flux[k - 2] += float((rho[cells] * u[d][cells] * sgn).sum()) * (1 if k == 2 else -1)
        diag = {"mass": float(rho.sum()), "flux_in": flux[0], "flux_out": flux[1],
                "max_u": float((u * u).sum(0).max().sqrt()), "n_nonfinite": 0, "time": e.time}
        diag = {k: torch.tensor(v, dtype=torch.float64) if isinstance(v, float) else v for k, v in diag.items()}
        nz, ny, nx = g.shape
        pts = _probes(g, seed)
        rank = torch.full((g.mask.size,), -1, dtype=torch.int64, device="cuda")
        rank[e.box] = torch.arange(e.n, device="cuda")
        at = rank[torch.from_numpy((pts[:, 0] * ny + pts[:, 1]) * nx + pts[:, 2]).cuda()]
        return {"rho": rho, "u": u, "diag": diag, "probes": torch.stack([rho[at], *u[:, at]], 1), "rho_mean": rho,
                "u_mean": u, "n": 1}
    if kind == "batch":
        out = []
        for k, g in enumerate(_members(case, seed)):
            e = _Exact(g, case, seed + k)
            e.step(case["steps"])
            out.append(e.fields())
        return out
    g = _geometry(case, seed)
    m = _mask(g)
    if kind == "corrector":
        rho, u, fm = _fine_snapshot(m, seed)
        nz, ny, nx = m.shape
        w = fm.double().reshape(nz, 2, ny, 2, nx, 2)
        k = w.sum((1, 3, 5))
        mean = [((f.double().reshape(nz, 2, ny, 2, nx, 2) * w).sum((1, 3, 5)) / k.clamp(min=1)) for f in (rho, *u)]
        crho, cu = mean[0], torch.stack(mean[1:])
        o = _net64(_params64(seed), crho, cu, m)
        return {"rho": crho, "u": cu, "du": DU_SCALE * o.clamp(-2, 2) * _bulk(m)}
    if kind == "train":
        rho, u, target = _pair(m, seed)
        bulk = _bulk(m).double()
        p = [v.requires_grad_(True) for v in _params64(seed)]
        mom = [(torch.zeros_like(v), torch.zeros_like(v)) for v in p]
        losses = []
        for t in range(1, case["steps"] + 1):
            r = (_net64(p, rho, u, m) - (target.double() - u.double()) / DU_SCALE) * bulk
            loss = (r * r).sum() / (3 * bulk.sum().clamp(min=1))
            grads = torch.autograd.grad(loss, p)
            losses.append(loss.detach())
            new = []
            for k, (v, gr) in enumerate(zip(p, grads)):
                a, b = 0.9 * mom[k][0] + 0.1 * gr, 0.999 * mom[k][1] + 0.001 * gr * gr
                mom[k] = a, b
                new.append((v.detach() - case["lr"] * (a / (1 - 0.9 ** t)) / ((b / (1 - 0.999 ** t)).sqrt() + 1e-8))
                           .requires_grad_(True))
            p = new
        return {"loss": losses, "params": torch.cat([v.detach().reshape(-1) for v in p])}
    e = _Exact(g, case, seed)
    e.step(case["steps"])
    rho, u = e.dense()
    o = _net64(_params64(seed), rho, u, m)
    e.correct(0.25 * (DU_SCALE / 10) * o.clamp(-2, 2) * _bulk(m))
    rho, u = e.dense()
    return {"rho": rho, "u": u}
