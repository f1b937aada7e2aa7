"""Performance cases of the cased-well simulator and its trace surrogate.

A case is one piece of work a user of the package has it do, through the public
Python layer: steps of one well (`Simulation`), of a batch of wells
(`BatchSimulation`), of a well on the azimuthally refined grid
(`RefinedSimulation`), predictions and training epochs of the trace surrogate
(`Surrogate`).  The handles live across passes, as in a user's program; a pass
advances them further and reads back what the program wants: the receiver
traces, and for one well the nine fields (`get_planes`, a snapshot).  Wells of
one handle start from smooth random velocities (a restart from a snapshot), so
that the whole grid carries waves, as it does for most of a real run's 6000 to
20000 steps; batches and refined wells start at rest, which is how their API
starts.

`exact` restates the scheme and the network in 64 bits with plain torch.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2302_13907_gb300 import workloads as W
from paper_2302_13907_gb300.binding import SURROGATE_DEFAULT, BatchSimulation, RefinedSimulation, Simulation, Surrogate

ELEM = {"f32": 4, "bf16": 2, "f16": 2, "f16sr": 2}
DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16, "f16sr": torch.float16}
IMPEDANCE = 1000.0 * 1500.0  # of the well's liquid, where every source sits: velocity scale of FP16 storage


# ------------------------------------------------------------------- the cases
def _well(name, nr, nth, nz, pml, d, steps, storage="f32", source="monopole", noise=False, watchdog=0):
    return dict(name=name, kind="well", nr=nr, nth=nth, nz=nz, pml=pml, d=d, steps=steps, storage=storage,
                source=source, noise=noise, watchdog=watchdog)


def listed():
    return [
        # a quick look at a short well on a coarse grid: small launches, everything in L2
        _well("short coarse well", 60, 16, 300, 10, 0.005, 256),
        # the 20 m well at full resolution with rock noise: the production run
        _well("20 m well", 180, 64, 8192, 16, 0.0025, 64, noise=True),
        # one cement-hardening case on its own (the plain solver behind the surrogate's data)
        _well("cement case", 120, 32, 3072, 16, 0.0025, 128),
        # a 20 m section of the realistic cased well (collars, two casings) with the torsion source: few azimuthal nodes
        _well("realistic section, torsion", 64, 8, 8000, 16, 0.0025, 192, source="torsion"),
        # sizes that nothing divides, a point force on the axis
        _well("ragged well, point force", 75, 22, 1501, 13, 0.0025, 256, source="transverse", noise=True),
        # the precision variants on the 2.56 m crop of the 20 m well, 16-bit storage
        _well("crop, BF16", 180, 64, 1024, 16, 0.0025, 128, storage="bf16", noise=True),
        # FP16 with stochastic rounding under the device watchdog
        _well("crop, FP16-SR, watchdog", 180, 64, 1024, 16, 0.0025, 64, storage="f16sr", noise=True, watchdog=16),
        # 64 miniature cement cases in one batch: one alone leaves most of the GPU idle
        dict(name="64 miniature wells", kind="batch", wells=64, nr=36, nth=8, nz_lo=240, nz_hi=240, pml=8, d=0.005,
             steps=256),
        # the 20 m well on the azimuthally refined grid
        dict(name="20 m well, refined", kind="refined", nr=180, nth=64, nz=8192, pml=16, d=0.0025, steps=64),
        # a reach crop of a cement case on the refined grid: what generates the surrogate's data, thousands of times
        dict(name="cement crop, refined", kind="refined", nr=120, nth=32, nz=1298, pml=16, d=0.0025, steps=256),
        # the surrogate answering a set of held-out cases from host arrays
        dict(name="surrogate, 512 answers", kind="predict", cases=512, batch=64),
        # one epoch of the surrogate's training on host arrays
        dict(name="surrogate, training epoch", kind="train", cases=256, batch=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["well", "well", "well", "well", "16 bit", "16 bit", "batch", "refined", "refined", "predict",
                       "train"])
    if kind == "predict":
        return dict(kind=kind, cases=_log(rng, 16, 512), batch=rng.choice([16, 32, 64]))
    if kind == "train":
        batch = rng.choice([16, 32, 64])
        return dict(kind=kind, cases=_log(rng, batch, 512), batch=batch)
    d = rng.choice([0.0025, 0.0025, 0.005])
    if kind == "batch":
        lo = _log(rng, 120, 400)
        return dict(kind=kind, wells=_log(rng, 4, 64), nr=rng.randint(34, 60), nth=2 * rng.randint(2, 8), nz_lo=lo,
                    nz_hi=lo + rng.randint(0, 200), pml=rng.randint(6, 12), d=0.005, steps=_log(rng, 64, 256))
    nr = rng.randint(66, 180) if d < 0.004 else rng.randint(34, 90)
    pml = rng.randint(8, 18)
    nz = _log(rng, 200, 8192)
    if kind == "refined":
        nth = rng.choice([16, 32, 64])
        cells = nth * (nr + pml) * nz
        return dict(kind=kind, nr=nr, nth=nth, nz=nz, pml=pml, d=d, steps=max(16, min(256, int(4e9 / cells))))
    nth = 2 * _log(rng, 2, 32)
    cells = nth * (nr + pml) * nz
    steps = max(16, min(256, int(4e9 / cells)))
    noise = rng.random() < 0.5
    if kind == "16 bit":
        c = _well("", nr, nth, nz, pml, d, min(steps, 128), storage=rng.choice(["bf16", "f16", "f16sr"]), noise=noise,
                  watchdog=rng.choice([0, 0, 16]))
    else:
        c = _well("", nr, nth, nz, pml, d, steps, noise=noise, watchdog=rng.choice([0, 0, 0, 32]),
                  source=rng.choice(["monopole", "monopole", "transverse", "longitudinal"]))
    del c["name"]
    return c


# ---------------------------------------------------------------------- inputs
def _smooth(gen, shape, coarse):
    """Smooth random values of `shape`, from normal deviates every `coarse` cells."""
    n = [max(2, -(-s // c) + 1) for s, c in zip(shape, coarse)]
    x = torch.randn([1, 1] + n, generator=gen, device="cuda")
    return F.interpolate(x, size=list(shape), mode="trilinear", align_corners=True)[0, 0]


def _add_rock_noise(med, gen):
    """+-5 % correlated perturbation of the rock's speeds, in steps of 1e-4 (workloads.Noise), drawn on the GPU."""
    g = med.grid
    i0 = int(np.argmax(g.r_centre() >= 0.15))
    amp, quantum = 0.05, 1e-4
    nq = int(round(amp / quantum))
    x = _smooth(gen, (g.nth, g.NR - i0, g.NZ), (8, max(1, int(0.1 / g.dr)), max(1, int(0.1 / g.dz))))
    q = torch.round(x * (nq / x.abs().max())).to(torch.int32) + (nq + med.n_mat)
    med.cell_id[:, i0:, :] = q.to(torch.int16).cpu().numpy().view(np.uint16)
    f = 1.0 + quantum * np.arange(-nq, nq + 1)
    med.rho = np.concatenate([med.rho, np.full(2 * nq + 1, W.ROCK[0])])
    med.vp = np.concatenate([med.vp, W.ROCK[1] * f])
    med.vs = np.concatenate([med.vs, W.ROCK[2] * f])


def _cased(u, grid, steps, source=W.SOURCE_MONOPOLE):
    """A cement-hardening well from six uniform deviates u: top depth, ramp, top shear fraction, casing, pulse, direction."""
    length = grid.nz * grid.dz
    z_top = (0.4 + 0.2 * u[0]) * length
    med = W.cased_well(grid, z_top=z_top, ramp=min(0.3, 0.2 * length) * u[1], top_frac=float(u[2]),
                       casing_t=0.008 + 0.004 * u[3])
    zs = max(0.05 * length, z_top - 0.075)
    return W.Scenario("well", med, W.Source(kind=source, z=zs, theta=float(u[5]), f0=8e3 * (0.9 + 0.2 * u[4])),
                      W.on_axis_receivers(np.maximum(0.0, zs - 0.015 * np.arange(1, 9))), steps=steps)


def _scenario(case, seed):
    """The well of a one-well case and its initial velocities [3][nth][NR][NZ]."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    u = np.random.default_rng(int(seed)).random(6)
    if case["source"] == "torsion":
        sc = W.realistic_well_section(z0=96.0 + 8.0 * u[0], length=case["nz"] * case["d"], nth=case["nth"],
                                      nr=case["nr"], pml_r=case["pml"], pml_z=case["pml"], dr=case["d"], dz=case["d"],
                                      f0=8e3 * (0.9 + 0.2 * u[4]), steps=case["steps"])
    else:
        g = W.Grid(nr=case["nr"], nth=case["nth"], nz=case["nz"], pml_r=case["pml"], pml_z=case["pml"], dr=case["d"],
                   dz=case["d"])
        kind = {"monopole": W.SOURCE_MONOPOLE, "transverse": W.SOURCE_TRANSVERSE,
                "longitudinal": W.SOURCE_LONGITUDINAL}[case["source"]]
        sc = _cased(u, g, case["steps"], kind)
    if case.get("noise"):
        _add_rock_noise(sc.medium, gen)
    v = torch.stack([_smooth(gen, sc.grid.shape, (2, 4, 8)) for _ in range(3)]) / IMPEDANCE
    v[0, :, 0, :] = 0.0  # v_r on the axis and v_z beyond the last half-node are not unknowns
    v[2, :, :, -1] = 0.0
    return sc, v


def _batch_wells(case, seed):
    r = np.random.default_rng(int(seed))
    out = []
    for _ in range(case["wells"]):
        nz = int(r.integers(case["nz_lo"], case["nz_hi"] + 1))
        g = W.Grid(nr=case["nr"], nth=case["nth"], nz=nz, pml_r=case["pml"], pml_z=case["pml"], dr=case["d"],
                   dz=case["d"])
        out.append(_cased(r.random(6), g, case["steps"]))
    return out


def _refined_well(case, seed):
    g = W.Grid(nr=case["nr"], nth=case["nth"], nz=case["nz"], pml_r=case["pml"], pml_z=case["pml"], dr=case["d"],
               dz=case["d"])
    return _cased(np.random.default_rng(int(seed)).random(6), g, case["steps"]), W.refinement_rows(g)


_ARCH = SURROGATE_DEFAULT
_LEN = _ARCH["l0"] * 2 ** (len(_ARCH["chans"]) - 1)


def _shapes():
    c, flat = _ARCH["chans"], _ARCH["l0"] * _ARCH["chans"][0]
    s = [(_ARCH["in_dim"], _ARCH["h1"]), (_ARCH["h1"],), (_ARCH["h1"], _ARCH["h2"]), (_ARCH["h2"],),
         (_ARCH["h2"], flat), (flat,)]
    for a, b in zip(c, c[1:]):
        s += [(a, b, 4), (b,)]
    return s + [(c[-1], _ARCH["out_ch"]), (_ARCH["out_ch"],)]


def _network(seed):
    """Weights as one vector, and the inputs' mean and scale."""
    r = np.random.default_rng([int(seed), 7])
    th = [r.standard_normal(s) / math.sqrt(s[0] * (2 if len(s) == 3 else 1)) if len(s) > 1
          else 0.05 * r.standard_normal(s) for s in _shapes()]
    mean = np.array([5.0, 0.25, 0.5, 0.01, 1700.0, 2300.0], np.float32)
    scale = np.array([2.0, 0.15, 0.3, 0.0012, 100.0, 130.0], np.float32)
    return np.concatenate([t.ravel() for t in th]).astype(np.float32), mean, scale


def _queries(case, seed):
    return np.stack([W.case_features(int(seed) % 100000 * 1000 + q) for q in range(case["cases"])]).astype(np.float32)


def _targets(case, seed):
    """Decaying wave trains of the size the traces have after normalisation."""
    r = np.random.default_rng([int(seed), 11])
    t = np.arange(_LEN, dtype=np.float32) / _LEN
    a = r.standard_normal((case["cases"], _ARCH["out_ch"], 3, 1)).astype(np.float32)
    f = (2 + 12 * r.random((case["cases"], _ARCH["out_ch"], 3, 1))).astype(np.float32)
    return np.ascontiguousarray((a * np.sin(2 * np.pi * f * t) * np.exp(-2 * t)).sum(axis=2), np.float32)


# ------------------------------------------------------------------ the passes
def prepare(case, seed):
    stream = torch.cuda.Stream()
    kind = case["kind"]
    if kind == "well":
        sc, v = _scenario(case, seed)
        s = Simulation(sc, storage=case["storage"], watchdog_every=case["watchdog"], stream=stream.cuda_stream)
        g = sc.grid
        planes = s.config()[0] not in (2, 3)  # plane copies: the paths that update one buffer set
        if planes and case["storage"] == "f32":
            torch.cuda.synchronize()
            s.put_planes(0, 0, g.NZ, v.reshape(3, g.nth * g.NR, g.NZ).contiguous())
            s.sync()
        else:
            for name, x in zip(("vr", "vp", "vz"), v):
                s.set_field(name, x.cpu().numpy())
        out = [torch.empty(n, g.nth * g.NR, g.NZ, dtype=DTYPE[case["storage"]], device="cuda") for n in (3, 6)]
        torch.cuda.synchronize()
        return dict(case=case, sim=s, stream=stream, out=out, nz=g.NZ, planes=planes)
    if kind == "batch":
        b = BatchSimulation(_batch_wells(case, seed), stream=stream.cuda_stream)
        return dict(case=case, sim=b, stream=stream)
    if kind == "refined":
        sc, rows = _refined_well(case, seed)
        return dict(case=case, sim=RefinedSimulation(sc, rows, stream=stream.cuda_stream), stream=stream)
    net = Surrogate(max_batch=case["batch"], seed=1, stream=stream.cuda_stream)
    th, mean, scale = _network(seed)
    net.set_params(th)
    net.set_normalization(mean, scale, 1.5)
    st = dict(case=case, net=net, stream=stream, X=_queries(case, seed), seed=int(seed))
    if kind == "train":
        st["Y"] = _targets(case, seed)
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "well":
        s, out = state["sim"], state["out"]
        s.step(case["steps"])
        if state["planes"]:
            s.get_planes(0, 0, state["nz"], out[0])
            s.get_planes(1, 0, state["nz"], out[1])
        else:
            names = ("vr", "vp", "vz", "srr", "spp", "szz", "srp", "spz", "srz")
            for q, name in enumerate(names):
                x = torch.from_numpy(s.field(name)).reshape(out[0].shape[1:])
                (out[0][q] if q < 3 else out[1][q - 3]).copy_(x)
        # 16-bit storage: the fields are the result (a receiver's samples are sums of three of their values)
        if case["storage"] != "f32":
            s.sync()
            return {"velocity": out[0], "stress": out[1]}
        return {"traces": s.traces(), "velocity": out[0], "stress": out[1]}
    if case["kind"] == "batch":
        b = state["sim"]
        b.run(case["steps"])
        return {"traces": np.stack([b.traces(c) for c in range(b.n)])}
    if case["kind"] == "refined":
        return {"traces": state["sim"].step(case["steps"]).traces()}
    if case["kind"] == "predict":
        return {"traces": state["net"].forward(state["X"])}
    loss = state["net"].train(state["X"], state["Y"], epochs=1, batch=case["batch"], lr=1e-3, seed=state["seed"])
    return {"loss": loss, "weights": state["net"].params()}


# ------------------------------------------------------------------- the floor
def _well_work(cells, elem, radial, ends, steps):
    """A step reads the nine fields, the IDs and the layers' memory variables (12 and 6 FP32 values a cell) and
    writes the fields and the memory variables; about 130 operations a cell."""
    return {"bytes": steps * (cells * (18 * elem + 2) + 8 * (12 * radial + 6 * ends)), "flops": 130.0 * steps * cells}


def work(case):
    kind = case["kind"]
    if kind in ("well", "refined", "batch"):
        n, nr, p = case["nth"], case["nr"], case["pml"]
        if kind == "batch":
            nz = (case["nz_lo"] + case["nz_hi"]) / 2 + 2 * p
            k = case["wells"]
            return _well_work(k * n * (nr + p) * nz, 4, k * n * p * nz, k * n * (nr + p) * 2 * p, case["steps"])
        nz = case["nz"] + 2 * p
        if kind == "well":
            return _well_work(n * (nr + p) * nz, ELEM[case["storage"]], n * p * nz, n * (nr + p) * 2 * p, case["steps"])
        rows = [0] + W.refinement_rows(W.Grid(nr, n, case["nz"], p, p, case["d"], case["d"])) + [nr + p]
        col = sum((b - a) * (n >> (len(rows) - 2 - m)) for m, (a, b) in enumerate(zip(rows, rows[1:])))
        return _well_work(col * nz, 4, n * p * nz, col * 2 * p, case["steps"])
    n, macs, length = case["cases"], 0, _ARCH["l0"]
    for s in _shapes():
        if len(s) == 2:
            macs += s[0] * s[1] * (length if s[0] == _ARCH["chans"][-1] and s[1] == _ARCH["out_ch"] else 1)
        elif len(s) == 3:
            macs += s[0] * s[1] * 4 * length
            length *= 2
    params = sum(int(np.prod(s)) for s in _shapes())
    io = 4 * n * (_ARCH["in_dim"] + _ARCH["out_ch"] * _LEN)
    if kind == "predict":
        return {"bytes": 2 * params + io, "flops": 2.0 * macs * n}
    steps = -(-n // case["batch"])
    return {"bytes": steps * 26 * params + io, "flops": 6.0 * macs * n}


# ------------------------------------------------- the same in 64 bits, plain torch
def _interp(n, half):
    """[2n][n]: trigonometric interpolation of n nodes to 2n (to the half-way nodes of both for half = 1)."""
    t = (torch.arange(2 * n)[:, None] - 2 * torch.arange(n)[None, :] - 0.5 * half).double() * (math.pi / n)
    s = 1 + torch.cos(0.5 * n * t)
    for m in range(1, n // 2):
        s = s + 2 * torch.cos(m * t)
    return (s / n).cuda()


def _ricker(t, f0):
    a = (math.pi * f0 * (t - 2 / f0)) ** 2
    return (1 - 2 * a) * math.exp(-a)


class _Zone:
    """One zone of rows i0 .. i1 - 1 with n azimuthal nodes: coefficients, fields, memory variables."""

    def __init__(self, ids, below, i0, sc, dt, n, mat):
        g = sc.grid
        self.n, self.i0, self.rows, self.g, dr = n, i0, ids.shape[1], g, g.dr
        self.dth = 2 * math.pi / n
        i = torch.arange(i0, i0 + self.rows, device="cuda", dtype=torch.float64)[None, :, None]
        self.inv_ri = torch.where(i > 0, 1 / (i.clamp(min=1) * dr), torch.zeros_like(i))
        self.inv_rh = 1 / ((i + 0.5) * dr)
        rho, lam, mu, imu = mat
        idm = torch.cat([ids[:, :1] if below is None else below, ids[:, :-1]], 1)
        nxt = lambda x: torch.roll(x, -1, 0)  # noqa: E731
        up = lambda x: torch.cat([x[..., 1:], x[..., -1:]], -1)  # noqa: E731
        rc, rm, qc, qm = rho[ids], rho[idm], imu[ids], imu[idm]
        self.c_vr, self.c_vp, self.c_vz = 2 * dt / (rm + rc), 2 * dt / (rc + nxt(rc)), 2 * dt / (rc + up(rc))
        self.m_rp = 4 * dt / (qm + qc + nxt(qm) + nxt(qc))
        self.m_rz = 4 * dt / (qm + qc + up(qm) + up(qc))
        self.m_pz = 4 * dt / (qc + nxt(qc) + up(qc) + up(nxt(qc)))
        self.lam, self.l2m = dt * lam[ids], dt * (lam[ids] + 2 * mu[ids])
        if i0 == 0:
            for c in (self.c_vr, self.m_rp, self.m_rz):
                c[:, 0] = 0
        for c in (self.c_vz, self.m_rz, self.m_pz):
            c[..., -1] = 0
        del idm, rc, rm, qc, qm
        self.f = {q: torch.zeros(ids.shape, dtype=torch.float64, device="cuda")
                  for q in ("vr", "vp", "vz", "srr", "spp", "szz", "srp", "spz", "srz")}
        self.psi = {}
        self.profiles(sc, dt)

    def profiles(self, sc, dt):
        g, al = self.g, math.pi * sc.source.f0
        vmax = float(sc.medium.vp.max())

        def ab(d):
            b = torch.exp(-(d + al) * dt)
            return torch.where(d > 0, d * (b - 1) / (d + al), torch.zeros_like(d)).cuda(), \
                torch.where(d > 0, b, torch.ones_like(d)).cuda()

        Lr, Lz = g.pml_r * g.dr, g.pml_z * g.dz
        d0r, d0z = (-3 * vmax * math.log(1e-3) / (2 * L) for L in (Lr, Lz))
        self.lay = max(0, min(self.rows, self.i0 + self.rows - g.nr))  # rows in the radial layer
        i = torch.arange(self.i0 + self.rows - self.lay, self.i0 + self.rows, dtype=torch.float64)[None, :, None]
        self.r, self.q = {}, {}
        for half in (0, 1):
            x, r = ((i + 0.5 * half - g.nr) * g.dr).clamp(min=0), (i + 0.5 * half) * g.dr
            self.r[half] = ab(d0r * (x / Lr) ** 2)
            self.q[half] = ab(d0r * x ** 3 / (3 * Lr * Lr) / r)
        k = torch.cat([torch.arange(g.pml_z), torch.arange(g.NZ - g.pml_z, g.NZ)]).double()
        self.zc = ab(d0z * (torch.maximum((g.pml_z - 0.5 - k) * g.dz, (k - (g.pml_z + g.nz - 0.5)) * g.dz).clamp(min=0) / Lz) ** 2)
        self.zh = ab(d0z * (torch.maximum((g.pml_z - 1.0 - k) * g.dz, (k + 1.0 - g.pml_z - g.nz) * g.dz).clamp(min=0) / Lz) ** 2)

    def stretch_r(self, key, D, ab):
        if self.lay:
            s = D[:, self.rows - self.lay:]
            p = self.psi.get(key)
            p = ab[0] * s if p is None else ab[1] * p + ab[0] * s
            self.psi[key] = p
            s += p
        return D

    def stretch_z(self, key, D, ab):
        pz = self.g.pml_z
        s = torch.cat([D[..., :pz], D[..., D.shape[-1] - pz:]], -1)
        p = self.psi.get(key)
        p = ab[0] * s if p is None else ab[1] * p + ab[0] * s
        self.psi[key] = p
        D[..., :pz] += p[..., :pz]
        D[..., D.shape[-1] - pz:] += p[..., pz:]
        return D

    def low(self, x, ghost):  # row i - 1
        return torch.cat([torch.zeros_like(x[:, :1]) if ghost is None else ghost[:, None], x[:, :-1]], 1)

    def high(self, x, ghost):  # row i + 1
        return torch.cat([x[:, 1:], torch.zeros_like(x[:, :1]) if ghost is None else ghost[:, None]], 1)

    def km(self, x):
        return torch.cat([torch.zeros_like(x[..., :1]), x[..., :-1]], -1)

    def kp(self, x):
        return torch.cat([x[..., 1:], torch.zeros_like(x[..., :1])], -1)

    def velocity(self, gh):
        f, dr, dz, dth = self.f, self.g.dr, self.g.dz, self.dth
        jm, jp = (lambda x: torch.roll(x, 1, 0)), (lambda x: torch.roll(x, -1, 0))
        a, b = self.low(f["srr"], gh["srr"]), self.low(f["spp"], gh["spp"])
        D = self.stretch_r("vr r", (f["srr"] - a) / dr, self.r[0])
        D += self.stretch_r("vr q", (0.5 * (f["srr"] + a) - 0.5 * (f["spp"] + b) + (f["srp"] - jm(f["srp"])) / dth) * self.inv_ri,
                            self.q[0])
        D += self.stretch_z("vr z", (f["srz"] - self.km(f["srz"])) / dz, self.zc)
        f["vr"] += self.c_vr * D
        a = self.high(f["srp"], gh["srp"])
        D = self.stretch_r("vp r", (a - f["srp"]) / dr, self.r[1])
        D += self.stretch_r("vp q", (a + f["srp"] + (jp(f["spp"]) - f["spp"]) / dth) * self.inv_rh, self.q[1])
        D += self.stretch_z("vp z", (f["spz"] - self.km(f["spz"])) / dz, self.zc)
        f["vp"] += self.c_vp * D
        a = self.high(f["srz"], gh["srz"])
        D = self.stretch_r("vz r", (a - f["srz"]) / dr, self.r[1])
        D += self.stretch_r("vz q", (0.5 * (a + f["srz"]) + (f["spz"] - jm(f["spz"])) / dth) * self.inv_rh, self.q[1])
        D += self.stretch_z("vz z", (self.kp(f["szz"]) - f["szz"]) / dz, self.zh)
        f["vz"] += self.c_vz * D

    def stress(self, gh):
        f, dr, dz, dth = self.f, self.g.dr, self.g.dz, self.dth
        jm, jp = (lambda x: torch.roll(x, 1, 0)), (lambda x: torch.roll(x, -1, 0))
        a = self.high(f["vr"], gh["vr"])
        err = self.stretch_r("err", (a - f["vr"]) / dr, self.r[1])
        epp = self.stretch_r("epp", ((f["vp"] - jm(f["vp"])) / dth + 0.5 * (f["vr"] + a)) * self.inv_rh, self.q[1])
        ezz = self.stretch_z("ezz", (f["vz"] - self.km(f["vz"])) / dz, self.zc)
        f["srr"] += self.l2m * err + self.lam * (epp + ezz)
        f["spp"] += self.l2m * epp + self.lam * (err + ezz)
        f["szz"] += self.l2m * ezz + self.lam * (err + epp)
        del err, epp, ezz
        a = self.low(f["vp"], gh["vp"])
        D = self.stretch_r("rp r", (f["vp"] - a) / dr, self.r[0])
        D += self.stretch_r("rp q", ((jp(f["vr"]) - f["vr"]) / dth - 0.5 * (f["vp"] + a)) * self.inv_ri, self.q[0])
        f["srp"] += self.m_rp * D
        D = self.stretch_z("rz z", (self.kp(f["vr"]) - f["vr"]) / dz, self.zh)
        D += self.stretch_r("rz r", (f["vz"] - self.low(f["vz"], gh["vz"])) / dr, self.r[0])
        f["srz"] += self.m_rz * D
        D = self.stretch_r("pz q", (jp(f["vz"]) - f["vz"]) / dth * self.inv_rh, self.q[1])
        D += self.stretch_z("pz z", (self.kp(f["vp"]) - f["vp"]) / dz, self.zh)
        f["spz"] += self.m_pz * D


def _march(sc, rows, steps, v=None):
    """FP64 run of a well on zones that start at `rows` (none: the uniform grid): zones, receiver traces [n][steps]."""
    g, med, src = sc.grid, sc.medium, sc.source
    ids = torch.from_numpy(med.cell_id.view(np.int16)).cuda().to(torch.int32) & 0xFFFF
    cut = [0] + list(rows) + [g.NR]
    M = len(cut) - 1
    n_of = [g.nth >> (M - 1 - m) for m in range(M)]
    vp = torch.from_numpy(med.vp).cuda()
    dt = math.inf
    sub = [ids[:: g.nth // n_of[m], cut[m]:cut[m + 1]] for m in range(M)]
    for m in range(M):
        c = torch.stack([vp[sub[m][:, q]].max() for q in range(sub[m].shape[1])]).cpu().numpy()
        r = (np.arange(cut[m], cut[m + 1]) + 0.5) * g.dr * 2 * math.pi / n_of[m]
        dt = min(dt, float((sc.cfl / (c * np.sqrt(1 / g.dr ** 2 + 1 / r ** 2 + 1 / g.dz ** 2))).min()))
    mu = med.rho * med.vs ** 2
    with np.errstate(divide="ignore"):
        mat = [torch.from_numpy(x).cuda() for x in (med.rho, med.rho * med.vp ** 2 - 2 * mu, mu, 1 / mu)]
    Z = [_Zone(sub[m], sub[m - 1][:, -1:].repeat_interleave(2, 0) if m else None, cut[m], sc, dt, n_of[m], mat)
         for m in range(M)]
    del ids, sub
    if v is not None:
        for q, name in enumerate(("vr", "vp", "vz")):
            Z[0].f[name].copy_(v[q])
    P = [[_interp(n_of[m], h) for h in (0, 1)] for m in range(M - 1)]
    half = {"vp", "srp", "spz"}

    def ghosts(m, below, above):
        gh = dict.fromkeys(below + above)
        for q in below if m else ():
            gh[q] = P[m - 1][q in half] @ Z[m - 1].f[q][:, -1]
        for q in above if m + 1 < M else ():
            gh[q] = 0.5 * P[m][q in half].T @ Z[m + 1].f[q][:, 0]
        return gh

    ks = round(src.z / g.dz) + g.pml_z
    kr = torch.tensor([int(round(z / g.dz)) + g.pml_z for z in sc.receivers.z], device="cuda")
    f0, z0, A, dr, dz = Z[0].f, Z[0], src.amplitude, g.dr, g.dz
    j = torch.arange(z0.n, device="cuda", dtype=torch.float64)
    out = []
    for n in range(steps):
        gh = [ghosts(m, ("srr", "spp"), ("srp", "srz")) for m in range(M)]
        for m in range(M):
            Z[m].velocity(gh[m])
        if src.kind == W.SOURCE_TRANSVERSE:  # c_vr = dt / mean density
            f0["vr"][:, 1, ks] += A * _ricker(n * dt, src.f0) * z0.c_vr[:, 1, ks] * 2 * torch.cos(j * z0.dth - src.theta) / \
                (z0.n * dr * dr * z0.dth * dz)
        elif src.kind == W.SOURCE_LONGITUDINAL:
            f0["vz"][:, 0, ks] += A * _ricker(n * dt, src.f0) * z0.c_vz[:, 0, ks] / (math.pi * dr * dr * dz)
        gh = [ghosts(m, ("vp", "vz"), ("vr",)) for m in range(M)]
        for m in range(M):
            Z[m].stress(gh[m])
        w = dt * A * _ricker((n + 0.5) * dt, src.f0)
        if src.kind == W.SOURCE_MONOPOLE:
            for q in ("srr", "spp", "szz"):
                f0[q][:, 0, ks] += w / (math.pi * dr * dr * dz)
        elif src.kind == W.SOURCE_TORSION:
            i, ih = int(round(src.r / dr)), int(math.floor(src.r / dr))
            f0["srp"][:, i, ks] += w / (2 * math.pi * i * dr * dr * dz)
            f0["spz"][:, ih, ks] += w / (2 * math.pi * (ih + 0.5) * dr * dr * dz)
        out.append(-(f0["srr"][:, 0, kr] + f0["spp"][:, 0, kr] + f0["szz"][:, 0, kr]).mean(0) / 3)
    return Z, torch.stack(out, 1)


def _net(th, X, n_up):
    """The network on normalised inputs: [cases][channels][samples]."""
    gelu = lambda x: 0.5 * x * (1 + torch.tanh(math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)))  # noqa: E731
    h = X
    for q in (0, 2, 4):
        h = gelu(h @ th[q] + th[q + 1])
    h = h.reshape(X.shape[0], _ARCH["l0"], -1).transpose(1, 2)
    for q in range(6, 6 + 2 * n_up, 2):
        h = gelu(F.conv_transpose1d(h, th[q], th[q + 1], stride=2, padding=1))
    return torch.einsum("bct,co->bot", h, th[-2]) + th[-1][:, None]


def _split(th):
    out, o = [], 0
    for s in _shapes():
        n = int(np.prod(s))
        out.append(th[o:o + n].reshape(s))
        o += n
    return out


def _train(case, seed, th, X, Y):
    """One epoch as sur_train states it: seeded shuffle, minibatches, Adam, cosine learning rate."""
    n, batch, mask, st = case["cases"], case["batch"], (1 << 64) - 1, int(seed)
    perm = list(range(n))
    for q in range(n - 1, 0, -1):
        st = (st + 0x9E3779B97F4A7C15) & mask
        z = ((st ^ (st >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        p = (z ^ (z >> 31)) % (q + 1)
        perm[q], perm[p] = perm[p], perm[q]
    steps, losses = -(-n // batch), []
    m, v = torch.zeros_like(th), torch.zeros_like(th)
    for t in range(steps):
        at = torch.tensor(perm[t * batch:(t + 1) * batch], device="cuda")
        w = th.detach().clone().requires_grad_()
        loss = ((_net(_split(w), X[at], len(_ARCH["chans"]) - 1) - Y[at]) ** 2).mean()
        loss.backward()
        m, v = 0.9 * m + 0.1 * w.grad, 0.999 * v + 0.001 * w.grad ** 2
        lr = 0.5e-3 * (1 + math.cos(math.pi * t / steps))
        th = th - lr * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
        losses.append(float(loss))
    return torch.tensor([sum(losses) / steps], dtype=torch.float64), th.cpu()


def exact(case, seed):
    with torch.backends.cudnn.flags(enabled=False):
        kind = case["kind"]
        if kind == "well":
            sc, v = _scenario(case, seed)
            Z, tr = _march(sc, [], case["steps"], v)
            f, g = Z[0].f, sc.grid
            vs = IMPEDANCE if case["storage"] in ("f16", "f16sr") else 1.0  # amplitude 1: stresses unscaled
            out = {"velocity": torch.stack([f[q] * vs for q in ("vr", "vp", "vz")]).reshape(3, -1, g.NZ)}
            out["stress"] = torch.stack([f[q] for q in ("srr", "spp", "szz", "srp", "spz", "srz")]).reshape(6, -1, g.NZ)
            if case["storage"] == "f32":
                out["traces"] = tr
            return out
        if kind == "batch":
            return {"traces": torch.stack([_march(sc, [], case["steps"])[1] for sc in _batch_wells(case, seed)])}
        if kind == "refined":
            sc, rows = _refined_well(case, seed)
            return {"traces": _march(sc, rows, case["steps"])[1]}
        th, mean, scale = _network(seed)
        X = torch.from_numpy((_queries(case, seed).astype(np.float64) - mean) / scale).cuda()
        th = torch.from_numpy(th).double().cuda()
        if kind == "predict":
            return {"traces": torch.cat([_net(_split(th), x, len(_ARCH["chans"]) - 1) * 1.5 for x in X.split(64)])}
        Y = torch.from_numpy(_targets(case, seed)).double().cuda() / 1.5
        loss, w = _train(case, seed, th, X, Y)
        return {"loss": loss, "weights": w}
