"""The work that is timed: what programs built on this library ask of it.

A case is one kind of simulation at one size.  A pass advances it by `steps`
time steps through `Lattice.step` (or `step_record`) and reads the fields of
every species back into device memory with `get_moments_dev`, the loop of a
program that runs and looks at its fields now and then; `nn_grad` is one
training pass of the learned Poisson start.  The simulation goes on from pass
to pass.  Fields are kept in single precision, the precision the library
steps in; velocities of 16-bit lattices, whose stochastically rounded
populations resolve them to about three digits, in half precision.

`exact` restates the scheme in 64 bits with plain torch operations.
"""

import math

import numpy as np
import torch

from paper_1507_04891_gb300 import lbm
from paper_1507_04891_gb300 import workloads as WL

STORAGE_BYTES = {"fp32": 4, "fp16": 2, "bf16": 2}


def listed():
    return [
        # bulk mutual diffusion of two neutral species on a small box: one
        # short kernel per step, latency and launches decide
        dict(name="neutral_binary_32", kind="neutral", nx=32, ny=32, nz=32, species=2,
             storage="fp32", schmidt=10.0, pair=False, steps=100),
        # four neutral species with a drag frequency for every pair, on a box
        # of odd extents
        dict(name="neutral_quaternary_odd", kind="neutral", nx=97, ny=61, nz=45, species=4,
             storage="fp32", schmidt=30.0, pair=True, steps=20),
        # the benchmark: charged ternary 128^3, spectral Poisson solve every
        # step, whole steps as graphs
        dict(name="ternary_128", kind="bulk", nx=128, ny=128, nz=128, storage="fp32",
             schmidt=1.0, poisson="fft", graph=True, record=False, steps=20),
        # the same with half the bytes per population
        dict(name="ternary_128_fp16", kind="bulk", nx=128, ny=128, nz=128, storage="fp16",
             schmidt=1.0, poisson="fft", graph=True, record=False, steps=20),
        # steps driven from the host (the default of the constructor), BF16,
        # a high Schmidt number
        dict(name="ternary_64_bf16_host", kind="bulk", nx=64, ny=64, nz=64, storage="bf16",
             schmidt=100.0, poisson="fft", graph=False, record=False, steps=20),
        # a run restarted from densities in device memory, every step's
        # diagnostics recorded: the Poisson start has no history yet
        dict(name="restart_record_64", kind="bulk", nx=128, ny=64, nz=64, storage="fp32",
             schmidt=1.0, poisson="fft", graph=True, record=True, steps=20),
        # bulk electrolyte on extents the spectral solver does not take:
        # multigrid without walls, odd coarse levels
        dict(name="ternary_odd_mg", kind="bulk", nx=90, ny=50, nz=75, storage="fp32",
             schmidt=10.0, poisson="mg", graph=False, record=False, steps=5),
        # charged slit under a field
        dict(name="slit_64", kind="slit", nx=64, ny=64, width=64, sigma=-0.01, debye=8.0,
             storage="fp32", schmidt=10.0, steps=50),
        # the thin slit of the transport sweeps, where thousands of short
        # steps are run
        dict(name="slit_32x8x50", kind="slit", nx=32, ny=8, width=50, sigma=-1e-4, debye=10.0,
             storage="fp32", schmidt=1000.0, steps=100),
        # the batched sweep: 64 slits of their own widths, charges and
        # Schmidt numbers in one lattice
        dict(name="slit_stack_64", kind="stack", nx=32, ny=32, count=64, wmin=16, wmax=128,
             widths=1237, storage="fp16", steps=10),
        # charged spheres, ternary electrolyte, multigrid every step
        dict(name="porous_128", kind="porous", n=128, storage="fp32", schmidt=1.0, steps=5),
        # forward and backward pass of the learned Poisson start
        dict(name="nn_grad_64", kind="nn", n=64, hidden=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["neutral", "bulk", "bulk", "slit", "stack", "porous", "nn"])
    storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
    sc = round(math.exp(rng.uniform(0.0, math.log(1000.0))), 3)
    if kind == "neutral":
        s = rng.randint(2, 4)
        return dict(kind=kind, nx=_log_int(rng, 20, 128), ny=_log_int(rng, 20, 128),
                    nz=_log_int(rng, 20, 128), species=s, storage=storage, schmidt=sc,
                    pair=s > 2 and rng.random() < 0.5, steps=20)
    if kind == "bulk":
        if rng.random() < 0.6:
            graph = rng.random() < 0.7
            return dict(kind=kind, nx=2 ** rng.randint(4, 7), ny=2 ** rng.randint(4, 7),
                        nz=rng.choice([2 ** rng.randint(4, 7), _log_int(rng, 16, 128)]),
                        storage=storage, schmidt=sc, poisson="fft", graph=graph,
                        record=graph and rng.random() < 0.3, steps=20)
        return dict(kind=kind, nx=_log_int(rng, 20, 100), ny=_log_int(rng, 20, 100),
                    nz=_log_int(rng, 20, 100), storage=storage, schmidt=sc, poisson="mg",
                    graph=False, record=False, steps=5)
    if kind == "slit":
        w = _log_int(rng, 14, 100)
        return dict(kind=kind, nx=2 ** rng.randint(3, 6), ny=2 ** rng.randint(3, 6), width=w,
                    sigma=-round(10.0 ** rng.uniform(-4.0, -2.5), 6), debye=round(0.125 * w, 3),
                    storage=storage, schmidt=sc, steps=50)
    if kind == "stack":
        return dict(kind=kind, nx=2 ** rng.randint(3, 5), ny=2 ** rng.randint(3, 5),
                    count=_log_int(rng, 4, 48), wmin=16, wmax=rng.randint(40, 128),
                    widths=rng.randrange(1 << 20), storage=storage, steps=10)
    if kind == "porous":
        return dict(kind=kind, n=_log_int(rng, 32, 120), storage=storage, schmidt=sc, steps=5)
    return dict(kind="nn", n=_log_int(rng, 20, 64), hidden=rng.choice([4, 6, 8, 16]))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
class _Inputs:
    """Plain description of a simulation: arrays in 64 bits on the host."""

    def __init__(self, n0, valence, shape, bjerrum=0.0, e_ext=(0.0, 0.0, 0.0), omega_drag=1.0,
                 omega_z=None, pair=None, solid=None, sigma=None, u0=None):
        self.n0, self.valence, self.shape = n0, list(valence), tuple(shape)
        self.bjerrum, self.e_ext = bjerrum, tuple(e_ext)
        self.omega_drag, self.omega_z, self.pair = omega_drag, omega_z, pair
        self.solid, self.sigma, self.u0 = solid, sigma, u0


def _drag_of(sc):
    """omega_drag of a Schmidt number at omega_visc = 1 (nu = 1/6)."""
    return 1.0 / (0.5 + 0.5 / sc)


def _slits(case, rng):
    """The slit workloads of a case, each with its charge drawn from the seed
    and ions perturbed by a tenth of a per cent."""
    if case["kind"] == "slit":
        wls = [WL.slit(nx=case["nx"], ny=case["ny"], width=case["width"],
                       sigma=case["sigma"] * rng.uniform(0.8, 1.0), debye=case["debye"],
                       e_field=1e-4, schmidt=case["schmidt"])]
    else:
        # widths of the case; Schmidt numbers and charges (the co-ions of the
        # narrowest slit stay positive) of the seed
        widths = np.random.default_rng([case["widths"], case["count"]]).integers(
            case["wmin"], case["wmax"] + 1, size=case["count"])
        wls = [WL.slit(nx=case["nx"], ny=case["ny"], width=int(w), sigma=rng.uniform(-0.012, -0.002),
                       debye=8.0, e_field=1e-4, schmidt=math.exp(rng.uniform(0.0, math.log(1000.0))))
               for w in widths]
    for w in wls:
        for s in (1, 2):
            d = w.n0[s] * rng.uniform(-1e-3, 1e-3, size=w.shape)
            w.n0[s] += d
            w.n0[0] -= d
    return wls


def _inputs(case, seed):
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 17])
    kind = case["kind"]
    if kind == "neutral":
        shape, S = (case["nz"], case["ny"], case["nx"]), case["species"]
        od = _drag_of(case["schmidt"])
        if S == 2:  # a sinusoidal concentration mode, as in the diffusion runs
            x = np.arange(case["nx"])
            a = 0.5 + 0.01 * np.sin(2 * np.pi * x / case["nx"] + rng.uniform(0, 2 * np.pi))
            a = a + rng.uniform(-1e-3, 1e-3, size=shape)
            return _Inputs(np.stack([a, 1.0 - a]), [0.0, 0.0], shape, omega_drag=od)
        n0 = 1.0 / S + rng.uniform(-0.02, 0.02, size=(S,) + shape)
        u0 = rng.uniform(-0.02, 0.02, size=(S, 3) + shape)
        pair = None
        if case["pair"]:
            m = rng.uniform(0.6, 0.95, size=(S, S))
            pair = 0.5 * (m + m.T)
        return _Inputs(n0, [0.0] * S, shape, omega_drag=od, pair=pair, u0=u0)
    if kind == "bulk":
        shape = (case["nz"], case["ny"], case["nx"])
        wl = WL.ternary_bulk(shape=shape, seed=seed & 0x7FFFFFFF)
        return _Inputs(wl.n0, wl.valence, shape, wl.bjerrum, omega_drag=_drag_of(case["schmidt"]))
    if kind in ("slit", "stack"):
        wls = _slits(case, rng)
        cat = lambda v: np.concatenate(v, axis=0)  # noqa: E731
        n0 = np.stack([cat([np.where(w.solid, 1.0, w.n0[s]) for w in wls]) for s in range(3)])
        om = np.concatenate([np.full(w.shape[0], _drag_of(w.schmidt)) for w in wls])
        return _Inputs(n0, wls[0].valence, n0.shape[1:], wls[0].bjerrum, wls[0].e_ext,
                       omega_drag=_drag_of(wls[0].schmidt), omega_z=om,
                       solid=cat([w.solid for w in wls]), sigma=cat([w.sigma for w in wls]))
    wl = WL.porous_spheres(n=case["n"], seed=seed & 0x7FFFFFFF)
    n0 = np.where(wl.solid[None], 1.0, wl.n0)
    return _Inputs(n0, wl.valence, wl.shape, wl.bjerrum, omega_drag=1.0 if kind == "nn" else
                   _drag_of(case["schmidt"]), solid=wl.solid, sigma=wl.sigma)


def _nn_inputs(case, seed):
    """Walls, parameters and a normalised residual for the learned start."""
    i = _inputs(case, seed)
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 23])
    c = case["hidden"]
    a1, a2 = math.sqrt(3.0 / 54.0), 0.1 * math.sqrt(3.0 / (27.0 * c))
    p = np.concatenate([a1 * rng.uniform(-1, 1, 54 * c), 0.01 * rng.uniform(-1, 1, c),
                        a2 * rng.uniform(-1, 1, 27 * c)]).astype(np.float32)
    x0 = np.where(i.solid, 0.0, rng.standard_normal(i.shape))
    x0 = (x0 / math.sqrt((x0 ** 2).sum() / (~i.solid).sum())).astype(np.float32)
    return i, p, x0


def prepare(case, seed):
    kind = case["kind"]
    if kind == "nn":
        i, p, x0 = _nn_inputs(case, seed)
        n = case["n"]
        lat = lbm.Lattice(n, n, n, 1, bjerrum=i.bjerrum, poisson="mg")
        lat.set_walls(i.solid, i.sigma)
        lat.nn_init(hidden=case["hidden"], seed=1)
        lat.nn_params(p)
        return {"case": case, "lat": lat, "x0": x0}
    if kind in ("slit", "stack"):
        wls = _slits(case, np.random.default_rng([seed & 0x7FFFFFFF, 17]))
        if kind == "stack":
            lat, _ = lbm.stack_slits(wls, storage=case["storage"], step_graph=True)
        else:
            w = wls[0]
            nz, ny, nx = w.shape
            lat = lbm.Lattice(nx, ny, nz, 3, omega_drag=_drag_of(case["schmidt"]),
                              bjerrum=w.bjerrum, e_ext=w.e_ext, storage=case["storage"],
                              poisson="fft", step_graph=True)
            lat.set_walls(w.solid, w.sigma)
            for s in range(3):
                lat.set_species(s, 1.0, w.valence[s], np.where(w.solid, 1.0, w.n0[s]))
    else:
        i = _inputs(case, seed)
        nz, ny, nx = i.shape
        lat = lbm.Lattice(nx, ny, nz, len(i.valence), omega_drag=i.omega_drag, bjerrum=i.bjerrum,
                          storage=case["storage"], poisson=case.get("poisson", "mg"),
                          step_graph=case.get("graph", False))
        if i.solid is not None:
            lat.set_walls(i.solid, i.sigma)
        if i.pair is not None:
            lat.set_drag_matrix(i.pair)
        for s in range(len(i.valence)):
            lat.set_species(s, 1.0, i.valence[s], i.n0[s], None if i.u0 is None else i.u0[s])
    state = {"case": case, "lat": lat, "stream": torch.cuda.ExternalStream(lat.stream),
             "n": torch.empty((lat.S,) + lat.shape, dtype=torch.float64, device="cuda"),
             "u": torch.empty((lat.S, 3) + lat.shape, dtype=torch.float64, device="cuda")}
    if case.get("record"):
        state["n0"] = torch.from_numpy(i.n0).cuda()
        state["valence"] = i.valence
    torch.cuda.synchronize()
    return state


def run(state):
    case, lat = state["case"], state["lat"]
    if case["kind"] == "nn":
        loss, grad = lat.nn_loss_grad(state["x0"])
        return {"loss": loss, "grad": grad}
    out = {}
    if case.get("record"):
        for s in range(lat.S):
            lat.set_species_dev(s, 1.0, state["valence"][s], state["n0"][s].data_ptr())
        out["record"] = lat.step_record(case["steps"])
    else:
        lat.step(case["steps"])
    for s in range(lat.S):
        lat.get_moments_dev(s, state["n"][s].data_ptr(), state["u"][s].data_ptr())
    with torch.cuda.stream(state["stream"]):
        out["n"] = state["n"].float()
        out["u"] = state["u"].float() if case["storage"] == "fp32" else state["u"].half()
    return out


def work(case):
    """Per step every population read and written once, the potential read
    and written once; per pass the populations read and the moments written
    once.  Operations: about 250 per species and node and step, the
    transforms or cycles of the Poisson solve about 100 per node."""
    kind = case["kind"]
    if kind in ("porous", "nn"):
        nodes, fluid = case["n"] ** 3, 0.8 * case["n"] ** 3
    elif kind == "slit":
        nodes = fluid = case["nx"] * case["ny"] * case["width"]
    elif kind == "stack":
        nodes = fluid = case["nx"] * case["ny"] * case["count"] * (case["wmin"] + case["wmax"]) // 2
    else:
        nodes = fluid = case["nx"] * case["ny"] * case["nz"]
    if kind == "nn":
        c = case["hidden"]
        return {"bytes": 4.0 * nodes + 8.0 * 82 * c, "flops": 2.0 * 27 * c * nodes * (3 + 4)}
    s = case.get("species", 3)
    pop = 19.0 * s * STORAGE_BYTES[case["storage"]] * fluid
    charged = kind != "neutral"
    step = 2 * pop + (16.0 * fluid if charged else 0.0)
    flops = 250.0 * s * fluid + (100.0 * fluid if charged else 0.0)
    return {"bytes": case["steps"] * step + pop + 16.0 * s * nodes, "flops": case["steps"] * flops}


# --------------------------------------------------------------------------
# the scheme in 64 bits
# --------------------------------------------------------------------------
_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1.0 / 3] + [1.0 / 18] * 6 + [1.0 / 36] * 12
_OPP = [0, 2, 1, 4, 3, 6, 5, 8, 7, 10, 9, 12, 11, 14, 13, 16, 15, 18, 17]


def _at(a, c):
    """a at r + c on the periodic lattice."""
    return torch.roll(a, (-c[2], -c[1], -c[0]), (-3, -2, -1))


def _dot(c, v):
    """c . v over the components c has."""
    t = 0.0
    for d in range(3):
        if c[d]:
            t = t + c[d] * v[d]
    return t


class _Poisson:
    """A psi = 4 pi l_B (rho + w - mean over the connected fluid) and grad psi."""

    def __init__(self, i, dev):
        self.k = 4.0 * math.pi * i.bjerrum
        self.shape = i.shape
        self.walls = i.solid is not None
        if not self.walls:
            lam = 0.0
            for ax, n in enumerate(i.shape):
                e = 2.0 - 2.0 * torch.cos(2 * math.pi * torch.arange(n, device=dev, dtype=torch.float64) / n)
                lam = lam + e.reshape([-1 if a == ax else 1 for a in range(3)])
            lam[0, 0, 0] = 1.0
            self.lam = lam
            return
        fluid = torch.from_numpy(~i.solid).to(dev)
        self.fluid = fluid
        self.open = [fluid & _at(fluid, _C[p]) for p in range(1, 7)]
        solid, cnt = ~fluid, torch.zeros(i.shape, device=dev, dtype=torch.float64)
        for p in range(1, 7):
            cnt += _at(fluid, _C[p])
        q = torch.from_numpy(i.sigma).to(dev)
        q = torch.where(solid & (cnt > 0), q / cnt.clamp(min=1.0), torch.zeros_like(q))
        self.qn = [torch.where(fluid & ~o, _at(q, _C[p]), torch.zeros_like(q))
                   for p, o in zip(range(1, 7), self.open)]
        self.w = sum(self.qn)
        lab = torch.arange(fluid.numel(), device=dev).reshape(i.shape)
        while True:
            new = lab
            for _ in range(16):
                for p, o in zip(range(1, 7), self.open):
                    new = torch.where(o, torch.minimum(new, _at(new, _C[p])), new)
            if torch.equal(new, lab):
                break
            lab = new
        _, inv = torch.unique(lab[fluid], return_inverse=True)
        self.lab, self.size = inv, torch.bincount(inv).double()
        self.psi = torch.zeros(i.shape, device=dev, dtype=torch.float64)

    def _centred(self, v):
        x = v[self.fluid]
        mean = torch.zeros_like(self.size).index_add_(0, self.lab, x) / self.size
        out = torch.zeros_like(v)
        out[self.fluid] = x - mean[self.lab]
        return out

    def _A(self, v):
        r = torch.zeros_like(v)
        for p, o in zip(range(1, 7), self.open):
            r += torch.where(o, v - _at(v, _C[p]), torch.zeros_like(v))
        return r

    def gradient(self, rho):
        if not self.walls:
            s = torch.fft.fftn(self.k * rho)
            s[0, 0, 0] = 0.0
            psi = torch.fft.ifftn(s / self.lam).real
            return [0.5 * (_at(psi, _C[p]) - _at(psi, _C[p + 1])) for p in (1, 3, 5)]
        s = self._centred(self.k * (rho + self.w))
        x = self.psi
        r = self._centred(s - self._A(x))
        d, rr, stop = r.clone(), (r * r).sum(), 1e-24 * float((s * s).sum())
        for it in range(20000):
            if it % 16 == 0:
                if float(rr) <= stop:
                    break
                r, d = self._centred(r), self._centred(d)  # rounding feeds the constants
            Ad = self._A(d)
            a = rr / (d * Ad).sum().clamp(min=1e-300)
            x = x + a * d
            r = r - a * Ad
            new = (r * r).sum()
            d = r + (new / rr.clamp(min=1e-300)) * d
            rr = new
        self.psi = x
        g = []
        for p in (1, 3, 5):
            up = torch.where(self.open[p - 1], _at(x, _C[p]) - x, self.k * self.qn[p - 1])
            dn = torch.where(self.open[p], x - _at(x, _C[p + 1]), -self.k * self.qn[p])
            g.append(torch.where(self.fluid, 0.5 * (up + dn), torch.zeros_like(x)))
        return g


def _exact_moments(i, steps):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    S, z, om = len(i.valence), i.valence, 1.0  # omega_visc = 1 throughout
    fluid = None if i.solid is None else torch.from_numpy(~i.solid).to(dev)
    n0 = torch.from_numpy(np.ascontiguousarray(i.n0)).to(dev)
    u0 = None if i.u0 is None else torch.from_numpy(i.u0).to(dev)
    zero = torch.zeros(i.shape, dtype=torch.float64, device=dev)

    def mask(v):
        return v if fluid is None else torch.where(fluid, v, zero)

    def phi(n, ua, p):
        a = _dot(_C[p], ua)
        return n * _W[p] * (1.0 + 3.0 * a + 4.5 * a * a - 1.5 * (ua[0] ** 2 + ua[1] ** 2 + ua[2] ** 2))

    f = torch.empty((S, 19) + tuple(i.shape), dtype=torch.float64, device=dev)
    for s in range(S):
        ua = [zero] * 3 if u0 is None else list(u0[s])
        for p in range(19):
            f[s, p] = mask(phi(n0[s], ua, p))
    poisson = _Poisson(i, dev) if i.bjerrum > 0 else None
    wd = i.omega_drag
    if i.omega_z is not None:
        wd = torch.from_numpy(i.omega_z).to(dev)[:, None, None]

    def moments():
        n = [f[s].sum(0) for s in range(S)]
        safe = [v if fluid is None else torch.where(fluid, v, torch.ones_like(v)) for v in n]
        u = [[sum(_C[p][d] * f[s, p] for p in range(1, 19) if _C[p][d]) / safe[s] for d in range(3)]
             for s in range(S)]
        return n, u, safe

    for _ in range(steps):
        n, u, safe = moments()
        tot = sum(safe)
        ub = [sum(n[s] * u[s][d] for s in range(S)) / tot for d in range(3)]
        e = [zero + i.e_ext[d] for d in range(3)]
        if poisson is not None:
            g = poisson.gradient(sum(z[s] * n[s] for s in range(S)))
            e = [e[d] - g[d] / 3.0 for d in range(3)]
        v = [[u[s][d] + 0.5 * z[s] * e[d] for d in range(3)] for s in range(S)]
        new = torch.empty_like(f)
        for s in range(S):
            F = []
            for d in range(3):
                drag = 0.0
                for b in range(S):
                    w = wd if i.pair is None else float(i.pair[s][b])
                    drag = drag - w * (n[b] / tot) * (v[s][d] - v[b][d])
                F.append(z[s] * e[d] + drag)
            Fu = sum(F[d] * ub[d] for d in range(3))
            for p in range(19):
                fc, uc = _dot(_C[p], F), _dot(_C[p], ub)
                gp = n[s] * _W[p] * (3.0 * fc + 9.0 * fc * uc - 3.0 * Fu)
                new[s, p] = (1.0 - om) * f[s, p] + om * phi(n[s], u[s], p) + gp
        for s in range(S):
            for p in range(19):
                back = (-_C[p][0], -_C[p][1], -_C[p][2])
                pulled = _at(new[s, p], back)
                if fluid is not None:
                    pulled = mask(torch.where(_at(fluid, back), pulled, new[s, _OPP[p]]))
                f[s, p] = pulled
        del new
    n, u, _ = moments()
    u = torch.stack([torch.stack([mask(c) for c in us]) for us in u])
    return torch.stack(n), u


def _exact_nn(case, seed):
    i, p, x0 = _nn_inputs(case, seed)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    c = case["hidden"]
    p = torch.from_numpy(p).to(dev).double().requires_grad_(True)
    fluid = torch.from_numpy(~i.solid).to(dev)
    x0 = torch.from_numpy(x0).to(dev).double()
    m = fluid.double()
    taps = [(o % 3 - 1, (o // 3) % 3 - 1, o // 9 - 1) for o in range(27)]
    y = torch.zeros_like(x0)
    xs = torch.stack([_at(x0, t) for t in taps])
    ms = torch.stack([_at(m, t) for t in taps])
    for k in range(c):
        w = p[54 * k:54 * k + 54].reshape(2, 27)
        h = torch.tanh(p[54 * c + k] + torch.tensordot(w[0], xs, 1) + torch.tensordot(w[1], ms, 1))
        w2 = p[55 * c + 27 * k:55 * c + 27 * k + 27]
        y = y + torch.tensordot(w2, torch.stack([_at(h, t) for t in taps]), 1)
    y = y * m
    r = x0.clone()
    for q in range(1, 7):
        r = r - torch.where(fluid & _at(fluid, _C[q]), y - _at(y, _C[q]), torch.zeros_like(y))
    loss = (r * r * m).sum() / (x0 * x0).sum()
    grad, = torch.autograd.grad(loss, p)
    return {"loss": float(loss.detach()), "grad": grad.detach()}


def exact(case, seed):
    if case["kind"] == "nn":
        return _exact_nn(case, seed)
    n, u = _exact_moments(_inputs(case, seed), case["steps"])
    return {"record": None, "n": n, "u": u} if case.get("record") else {"n": n, "u": u}
