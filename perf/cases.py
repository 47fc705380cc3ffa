"""What a user of this framework has it do, as measurable cases.

Two kinds of work make up its use.  The FDTD solve of a zone (or of all zones
of a lens): a forward run, or the forward and adjoint runs of one topology
optimisation iteration.  And the U-Net surrogate: inference, the gradient of a
training batch, and the surrogate ascent of a warm start.  `listed` names one
case per regime, from runs whose time is launches and latency to the wide zone
that lives in HBM; `draw` gives others of the same ranges.

`exact` restates the physics and the network in 64-bit torch, from the
equations alone.

Focal phasors are returned as complex64: they are sums of single-precision
field DFTs and carry that precision, whatever type the binding hands out.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2501_07979_gb300 import Zone
from paper_2501_07979_gb300.lens import Lens
from paper_2501_07979_gb300.surrogate import Surrogate
from paper_2501_07979_gb300.warmstart import WarmStart
from zda_inputs import (ZoneSpec, focal_from_na, lens_zones, rho_for, smoothed_rho, zone_cfg1, zone_cfg2, zone_lwir,
                        zone_patch, zone_tiny, zone_visible)

DEV = "cuda:0"
FLOPS_PER_CELL_STEP = 96          # six complex components: two differences, two scalings, one update each
STATE_BYTES = 48                  # six complex FP32 components
L2_BYTES = 129e6


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the small zone of optimisation tests and of the 16-pixel warm start: every step is launch latency
        {"name": "tiny zone iteration", "kind": "zone", "zone": "tiny", "steps": 600, "run": "iteration"},
        # odd sizes in every direction (odd n_z: no vector path), three wavelengths, filter and projection
        {"name": "odd zone iteration", "kind": "zone", "zone": "odd", "steps": 250, "run": "iteration"},
        # the single-zone workload: one forward solve, its monitor field and its final fields read out
        {"name": "single zone forward", "kind": "zone", "zone": "cfg1", "steps": 1000, "run": "forward"},
        # the innermost zone of a lens, continuously axisymmetric, with the axis inside
        {"name": "axis zone iteration", "kind": "zone", "zone": "axis", "steps": 900, "run": "iteration"},
        # the zone size that the surrogate is trained and judged on (128 x 128 design pixels)
        {"name": "patch zone iteration", "kind": "zone", "zone": "patch", "steps": 830, "run": "iteration"},
        # zone 16 of the long-wave infrared lens: few phi cells, many radii, state about the size of L2
        {"name": "LWIR zone iteration", "kind": "zone", "zone": "lwir", "steps": 1600, "run": "iteration"},
        # zone 16 of the visible RGB lens: three wavelengths, a thick design layer, so DFTs weigh more
        {"name": "RGB zone iteration", "kind": "zone", "zone": "rgb", "steps": 1000, "run": "iteration"},
        # the wide zone of the headline benchmark (15 M cells) at a 10-wavelength arc: the field state in HBM
        {"name": "wide zone iteration", "kind": "zone", "zone": "wide", "steps": 600, "run": "iteration"},
        # a small lens: zones of uneven widths and folds, the axis zone among them, one graph per run
        {"name": "lens iteration", "kind": "lens", "zones": 6, "n_phi": 96, "n_z": 160, "time": 6.5, "zone_seed": 4},
        # surrogate inference over a data set
        {"name": "surrogate forward", "kind": "surrogate", "run": "forward", "batch": 256, "height": 128, "width": 128,
         "out_ch": 24},
        # the gradient of one training batch (the Adam update that follows is a sign for a first step, so
        # the gradients themselves are what can be compared)
        {"name": "surrogate gradient", "kind": "surrogate", "run": "gradient", "batch": 64, "height": 128,
         "width": 128, "out_ch": 24},
        # one step of the warm start: focal intensity of the surrogate's field and its gradient, one sample
        {"name": "surrogate ascent step", "kind": "ascent", "pixels": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["zone", "zone", "zone", "zone", "zone", "axis", "lens", "surrogate", "surrogate", "ascent"])
    if kind == "zone":
        n_z = rng.randrange(40, 161)
        c = {"kind": "zone", "zone": "any", "n_r": _log_int(rng, 24, 320), "n_phi": _log_int(rng, 4, 320), "n_z": n_z,
             "dr": rng.choice([0.1, 0.05, 0.05, 0.05, round(1 / 36, 6), 0.02]), "r_lo": round(math.exp(rng.uniform(math.log(5), math.log(400))), 3),
             "aspect": round(rng.uniform(0.4, 1.2), 3), "pml": rng.choice([5, 6, 8, 8, 8]),
             "wavelengths": rng.choice([1, 1, 2, 3, 3]), "time": round(rng.uniform(6.5, 9.0), 2),
             "filtered": rng.random() < 0.7, "radial_pml": 1 if rng.random() < 0.2 else 0,
             "run": rng.choice(["iteration", "iteration", "forward"])}
        if rng.random() < 0.5:
            c["n_z"] = n_z - n_z % 2
        while cost(c) > 0.8 * cost(listed()[7]):
            c["n_r"] = max(24, int(c["n_r"] * 0.7))
            c["n_phi"] = max(4, int(c["n_phi"] * 0.8))
        return c
    if kind == "axis":
        return {"kind": "zone", "zone": "axis", "n_r": _log_int(rng, 60, 300), "n_z": rng.randrange(100, 181),
                "steps": rng.randrange(700, 1100), "run": rng.choice(["iteration", "forward"])}
    if kind == "lens":
        return {"kind": "lens", "zones": rng.randrange(3, 7), "n_phi": rng.randrange(16, 97), "n_z": 2 * rng.randrange(50, 81),
                "time": round(rng.uniform(6.0, 6.5), 2), "zone_seed": rng.randrange(1000)}
    if kind == "surrogate":
        run_ = rng.choice(["forward", "gradient"])
        return {"kind": "surrogate", "run": run_, "batch": _log_int(rng, 1, 256 if run_ == "forward" else 64),
                "height": 8 * rng.randrange(2, 17), "width": 8 * rng.randrange(2, 17), "out_ch": 4 * rng.randrange(1, 8)}
    return {"kind": "ascent", "pixels": 8 * rng.randrange(2, 17)}


# ------------------------------------------------------------------ workload descriptions
def _dt(s):
    if s.n_fold == 0:
        mid = (s.m / (s.r_lo if s.r_lo > 0 else 0.5 * s.dr)) ** 2
    else:
        mid = 1.0 / (s.r_lo * 2 * math.pi / s.n_fold / s.n_phi) ** 2
    return s.courant / math.sqrt(1 / s.dr ** 2 + mid + 1 / s.dz ** 2)


def _spec(c):
    """The zone description of a zone case."""
    z, n = c["zone"], c.get("steps", 1)
    if z == "tiny":
        return zone_tiny(n_steps=n)
    if z == "odd":
        return zone_tiny(n_r=27, n_phi=7, n_z=45, pml_r_in=3, pml_r_out=5, pml_z=5, n_steps=n, layer_k0=(0, 15, 19),
                         design_k0=15, design_k1=19, source_k=8, monitor_k=26, wavelengths=(0.85, 1.0, 1.2),
                         filter_radius=0.2, beta=3.0, pulse_sigma=0.4, pulse_t0=1.6)
    if z == "cfg1":
        return dataclasses.replace(zone_cfg1(), n_steps=n)
    if z == "axis":
        s = dataclasses.replace(lens_zones()[0], n_steps=n)
        return dataclasses.replace(s, n_r=c.get("n_r", s.n_r), n_z=c.get("n_z", s.n_z), focal=40.0)
    if z == "patch":
        return zone_patch(200.0, n)
    if z == "lwir":
        return zone_lwir(16, n)
    if z == "rgb":
        return zone_visible(16, "rgb", n)
    if z == "wide":      # arc of 10 wavelengths, as the zones of the lens workload have
        return dataclasses.replace(zone_cfg2(n), n_fold=126)
    k0 = int(round(0.3 * c["n_z"]))
    k1 = k0 + max(3, int(round(0.09 * c["n_z"])))
    lams = {1: (1.0,), 2: (0.9, 1.1), 3: (0.82, 1.0, 1.18)}[c["wavelengths"]]
    fold = max(1, int(round(2 * math.pi * c["r_lo"] / (c["n_phi"] * c["aspect"] * c["dr"]))))
    s = ZoneSpec(r_lo=c["r_lo"], n_r=c["n_r"], n_phi=c["n_phi"], n_z=c["n_z"], n_fold=fold, dr=c["dr"], dz=c["dr"],
                 pml_r_in=c["pml"], pml_r_out=c["pml"], pml_z=c["pml"], layer_k0=(0, k0, k1), layer_eps=(2.1, 1.0, 1.0),
                 design_k0=k0, design_k1=k1, eps_lo=1.0, eps_hi=5.76, source_k=c["pml"] + 3,
                 monitor_k=min(k1 + max(4, int(0.1 * c["n_z"])), c["n_z"] - c["pml"] - 2),
                 filter_radius=1.6 * c["dr"] if c["filtered"] else 0.0, beta=8.0 if c["filtered"] else 0.0,
                 wavelengths=lams, pulse_sigma=0.4, pulse_t0=1.6, focal=1.5 * c["r_lo"])
    return dataclasses.replace(s, n_steps=int(math.ceil(c["time"] / _dt(s))))


def _lens_specs(c):
    """Uneven zones from the axis out; each runs the same simulated time."""
    specs = lens_zones(c["zones"], 10.0 * c["zones"], seed=c["zone_seed"], n_phi=c["n_phi"], n_z=c["n_z"], n_steps=1)
    f = focal_from_na(10.0 * c["zones"], 0.3)
    return [dataclasses.replace(s, n_steps=int(math.ceil(c["time"] / _dt(s))), focal=f) for s in specs]


def _patch(c):
    return zone_patch(200.0, 830, n_design=c["pixels"], n_phi=c["pixels"], arc=0.05 * c["pixels"])


def _specs(c):
    return _lens_specs(c) if c["kind"] == "lens" else [_spec(c)]


def cost(c):
    """Cell updates of a zone or lens case."""
    return sum(s.cells * s.n_steps for s in _specs(c)) * (1 if c.get("run") == "forward" else 2)


def _layers(in_ch, out_ch):
    """(kernel, inputs, outputs, level) of the U-Net's convolutions in parameter order."""
    enc = [(3, in_ch if l == 0 and not b else 64, 64, l) for l in range(3) for b in range(2)]
    dec = [(3, 64 if b else 128, 64, l) for l in (2, 1, 0) for b in range(2)]
    return enc + [(3, 64, 64, 3), (3, 64, 64, 3)] + dec + [(1, 64, out_ch, 0)]


def work(case):
    if case["kind"] in ("surrogate", "ascent"):
        if case["kind"] == "ascent":
            b, h, w, co, run_ = 1, case["pixels"], case["pixels"], 24, "gradient"
        else:
            b, h, w, co, run_ = case["batch"], case["height"], case["width"], case["out_ch"], case["run"]
        layers = _layers(1, co)
        flops = sum(2.0 * b * (h >> l) * (w >> l) * k * k * ci * o for k, ci, o, l in layers)
        params = sum(k * k * ci * o + o for k, ci, o, _ in layers)
        pix = b * h * w
        if run_ == "forward":
            return {"bytes": 4.0 * (pix * (1 + co) + params), "flops": flops}
        return {"bytes": 4.0 * (pix * (1 + 2 * co) + 2 * params), "flops": 3 * flops}
    total = {"bytes": 0.0, "flops": 0.0}
    runs = 1 if case.get("run") == "forward" else 2
    for s in _specs(case):
        pixels, q = s.n_r_design * s.n_phi, 2 * len(s.wavelengths)
        out = 8.0 * 2 * q * s.n_r * s.n_phi + (STATE_BYTES * s.cells if case.get("run") == "forward" else 4.0 * pixels)
        # a state that fits on the chip need not leave it between steps; one that does not is read and
        # written once a step
        moved = 2.0 * STATE_BYTES * s.cells * s.n_steps * runs if STATE_BYTES * s.cells > L2_BYTES else 0.0
        total["bytes"] += 4.0 * pixels + out + moved
        total["flops"] += float(FLOPS_PER_CELL_STEP) * s.cells * s.n_steps * runs
    return total


# ------------------------------------------------------------------ inputs and runs
def _rho(spec, seed):
    return torch.tensor(rho_for(spec, seed), dtype=torch.float32, device=DEV)


def _net_params(case, seed):
    """He-normal weights with a tenth of that in the head, small biases; the layout the network documents."""
    rng = np.random.default_rng(seed)
    co = case.get("out_ch", 24)
    parts = []
    for n, (k, ci, o, _) in enumerate(_layers(1, co)):
        std = math.sqrt(2.0 / (k * k * ci)) * (0.1 if n == 14 else 1.0)
        parts += [rng.standard_normal(o * k * k * ci) * std, rng.standard_normal(o) * 0.02]
    return np.concatenate(parts).astype(np.float32)


def _net_data(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    shape = (case["batch"], case["height"], case["width"])
    x = torch.rand((*shape, 1), generator=g, device=DEV)
    return x, torch.randn((*shape, case["out_ch"]), generator=g, device=DEV) if case["run"] == "gradient" else None


def prepare(case, seed):
    if case["kind"] == "zone":
        spec = _spec(case)
        zone = Zone(spec)
        if case.get("radial_pml"):
            zone.set_radial_pml(1)
        return {"case": case, "zone": zone, "rho": _rho(spec, seed)}
    if case["kind"] == "lens":
        specs = _lens_specs(case)
        return {"case": case, "lens": Lens([Zone(s) for s in specs]), "rho": [_rho(s, seed + 100 * i) for i, s in enumerate(specs)]}
    if case["kind"] == "ascent":
        spec = _patch(case)
        ws = WarmStart(spec, batch=1)
        ws.scale = 0.25
        ws.net.set_params(_net_params(case, seed))
        return {"case": case, "ws": ws, "rho": torch.tensor(smoothed_rho(spec.n_r_design, spec.n_phi, seed, mode="minmax"), dtype=torch.float32, device=DEV)}
    net = Surrogate(case["height"], case["width"], 1, case["out_ch"], case["batch"])
    net.set_params(_net_params(case, seed))
    x, target = _net_data(case, seed)
    return {"case": case, "net": net, "x": x, "target": target}


def _c64(S):
    return np.asarray(S).astype(np.complex64)


def run(state):
    case = state["case"]
    if case["kind"] == "zone":
        zone = state["zone"]
        if case["run"] == "forward":
            S = zone.forward(state["rho"])
            return {"S": _c64(S), "monitor": zone.monitor_dft(), "fields": zone.fields()}
        value, grad = zone.iteration(state["rho"])
        return {"I": value, "grad": grad, "monitor": zone.monitor_dft()}
    if case["kind"] == "lens":
        lens = state["lens"]
        S = lens.forward(state["rho"])
        grads = lens.adjoint(4.0 * S)
        return {"S": _c64(S), "grads": grads}
    if case["kind"] == "ascent":
        value, grad = state["ws"].surrogate_value_and_grad(state["rho"])
        return {"I": value, "grad": grad}
    net = state["net"]
    y = net.forward(state["x"])
    if case["run"] == "forward":
        return {"y": y}
    loss, dy = net.mse(y, state["target"])
    net.backward(dy)
    return {"loss": loss, "grads": net.grads()}


# ------------------------------------------------------------------ the same in 64 bits
F64, C128 = torch.float64, torch.complex128


def _t(x, dtype=F64):
    return torch.as_tensor(np.asarray(x), dtype=dtype, device=DEV)


def _shift(F, axis, by):
    """F at index + by along an axis, zero outside (the walls behind the PMLs conduct perfectly)."""
    out = torch.zeros_like(F)
    n = F.shape[axis]
    if by > 0:
        out.narrow(axis, 0, n - 1).copy_(F.narrow(axis, 1, n - 1))
    else:
        out.narrow(axis, 1, n - 1).copy_(F.narrow(axis, 0, n - 1))
    return out


class _Solver:
    """The Bloch-reduced Yee scheme of one wedge, convolutional PMLs, running DFTs, discrete adjoint."""

    def __init__(self, s, radial_pml):
        self.s, self.metric = s, bool(radial_pml)
        self.bor = s.n_fold == 0
        self.tau = 2 * math.pi / (1 if self.bor else s.n_fold)
        self.dphi = self.tau / s.n_phi
        self.dt = _dt(s)
        lam = np.asarray(s.wavelengths, float)
        self.w = np.concatenate([2 * np.pi / lam, -2 * np.pi / lam])
        self.i0, self.i1 = s.pml_r_in, s.n_r - s.pml_r_out
        self.nk = s.design_k1 - s.design_k0 + 1
        self.rn, self.rh = s.r_lo + np.arange(s.n_r) * s.dr, s.r_lo + (np.arange(s.n_r) + 0.5) * s.dr
        with np.errstate(divide="ignore"):
            self.irn = np.where(self.rn > 0, 1.0 / self.rn, 0.0)
        self.irh = 1.0 / self.rh
        r_end, z_end = s.r_lo + s.n_r * s.dr, s.n_z * s.dz
        zn, zh = np.arange(s.n_z) * s.dz, (np.arange(s.n_z) + 0.5) * s.dz
        self.cr_n, self.cr_h = (self._pml(x, s.r_lo, r_end, s.pml_r_in, s.pml_r_out, s.dr, self.metric) for x in (self.rn, self.rh))
        self.cz_n, self.cz_h = (self._pml(x, 0.0, z_end, s.pml_z, s.pml_z, s.dz, False) for x in (zn, zh))
        j = np.arange(s.n_phi)
        m = 0 if self.bor else s.m
        self.ph_n, self.ph_h = np.exp(1j * m * j * self.dphi), np.exp(1j * m * (j + 0.5) * self.dphi)
        self.n = np.arange(s.n_steps)
        self.tw = np.exp(1j * self.w[None] * ((self.n + 1) * self.dt)[:, None]) * self.dt
        zf = s.focal - (s.monitor_k - s.design_k1) * s.dz
        top = math.sqrt([e for k, e in zip(s.layer_k0, s.layer_eps) if s.monitor_k >= k][-1])
        kk = 2 * np.pi * top / np.tile(lam, 2)
        fold = 1 if self.bor else s.n_fold

        def kern(r):
            R = np.sqrt(zf ** 2 + r ** 2)[None]
            K = (zf / R) * (1 / R - 1j * kk[:, None]) * np.exp(1j * kk[:, None] * R) / R / (2 * np.pi)
            return 0.5 * fold * K * r[None] * self.dphi
        i = np.arange(s.n_r)
        wr = np.where((i >= self.i0) & (i < self.i1), s.dr, 0.0)
        wp = np.where((i >= self.i0) & (i <= self.i1), s.dr, 0.0) * np.where((i == self.i0) | (i == self.i1), 0.5, 1.0)
        self.Gr, self.Gp = kern(self.rh) * wr, kern(self.rn) * wp
        q = len(lam)
        self.Gr[q:], self.Gp[q:] = self.Gr[q:].conj(), self.Gp[q:].conj()
        self.Gp = -1j * self.Gp
        self.wt = 2 / self.dt * np.sin(self.w * self.dt / 2)

    def _pml(self, pos, lo, hi, n_in, n_out, h, stretched):
        """b, c of the derivative's recursion and bm, cm of the stretched radius' (zero: real radius)."""
        s = self.s
        a_max = 0.1 * math.pi * s.pulse_f0
        out = np.zeros((4, pos.size))
        for t, x0 in enumerate(pos):
            x, thick, outer = 0.0, h, False
            if n_in > 0 and x0 < lo + n_in * h:
                thick = n_in * h
                x = (lo + thick - x0) / thick
            if n_out > 0 and x0 > hi - n_out * h:
                thick, outer = n_out * h, True
                x = (x0 - (hi - thick)) / thick
            x = min(max(x, 0.0), 1.0)
            if x <= 0:
                continue
            smax = -2.0 * math.log(1e-8) / thick
            sg, al = smax * x ** 3, a_max * (1 - x)
            if stretched and outer:
                al = a_max
                sm = smax * thick * x ** 4 / 4 / x0
                out[2, t] = math.exp(-(sm + al) * self.dt)
                out[3, t] = sm / (sm + al) * (out[2, t] - 1)
            out[0, t] = math.exp(-(sg + al) * self.dt)
            out[1, t] = sg / (sg + al) * (out[0, t] - 1)
        return out

    # ---- density
    def tilde(self, rho):
        s = self.s
        x = rho
        if s.filter_radius > 0:
            R = s.filter_radius
            rc = _t(s.r_lo + (self.i0 + 0.5 + np.arange(s.n_r_design)) * s.dr)[:, None]
            di_max = min(int(R / s.dr), s.n_r_design - 1)
            dj_max = int(R / ((s.r_lo + (self.i0 + 0.5) * s.dr) * self.dphi))
            num, den = torch.zeros_like(x), torch.zeros_like(rc)
            rows = torch.arange(s.n_r_design, device=DEV)
            for di in range(-di_max, di_max + 1):
                ok = ((rows + di >= 0) & (rows + di < s.n_r_design))[:, None]
                src = x[(rows + di).clamp(0, s.n_r_design - 1)]
                for dj in range(-dj_max, dj_max + 1):
                    wgt = (1 - torch.sqrt((di * s.dr) ** 2 + (rc * dj * self.dphi) ** 2) / R).clamp(min=0) * ok
                    num = num + wgt * torch.roll(src, -dj, 1)
                    den = den + wgt
            x = num / den
        if s.beta > 0:
            b, e = s.beta, s.eta
            x = (math.tanh(b * e) + torch.tanh(b * (x - e))) / (math.tanh(b * e) + math.tanh(b * (1 - e)))
        return x

    def bars(self, rho):
        """Transverse density averages at the E_r, E_phi and E_z sites."""
        s = self.s
        full = torch.nn.functional.pad(self.tilde(rho), (0, 0, s.pml_r_in, s.pml_r_out))
        jm = torch.roll(full, 1, 1)
        im = torch.cat([full[:1], full[:-1]])
        jim = torch.roll(im, 1, 1)
        return 0.5 * (jm + full), 0.5 * (im + full), 0.25 * (jim + im + jm + full)

    def eps_tables(self):
        s = self.s
        k = np.arange(s.n_z)
        des = ((k >= s.design_k0) & (k < s.design_k1)).astype(float)
        base = np.array([[e for k0, e in zip(s.layer_k0, s.layer_eps) if kk >= k0][-1] for kk in k])
        base = np.where(des > 0, s.eps_lo, base)
        km = np.maximum(k - 1, 0)
        de = s.eps_hi - s.eps_lo
        return [_t(v) for v in (0.5 * (base[km] + base), 0.5 * de * (des[km] + des), base, de * des)]

    # ---- time loop
    def loop(self, inv_eps, src_k, src_r, src_p, mon_k):
        """src_r, src_p: step -> [n_r, n_phi] current at plane src_k.  Returns monitor and design DFTs and fields."""
        s, dt = self.s, self.dt
        shape = (s.n_r, s.n_phi, s.n_z)
        Er, Ep, Ez, Hr, Hp, Hz = (torch.zeros(shape, dtype=C128, device=DEV) for _ in range(6))
        bloch = complex(np.exp(1j * s.m * self.tau))
        zsl = [slice(0, s.pml_z), slice(s.n_z - s.pml_z, s.n_z)] if s.pml_z else []
        rsl = [x for x in (slice(0, s.pml_r_in), slice(s.n_r - s.pml_r_out, s.n_r)) if x.stop > x.start]
        irn, irh = _t(self.irn)[:, None, None], _t(self.irh)[:, None, None]
        Q = len(self.w)
        psi = {}

        def stretch(name, D, axis, table):
            """Adds the recursive convolution to a derivative inside its slabs, in place."""
            for n, sl in enumerate(zsl if axis == 2 else rsl):
                at = (slice(None), slice(None), sl) if axis == 2 else (sl,)
                b, c = (_t(v)[sl] if axis == 2 else _t(v)[sl][:, None, None] for v in table[:2])
                key = (name, n)
                if key not in psi:
                    psi[key] = [torch.zeros_like(D[at]), b, c]
                P, b, c = psi[key]
                P.mul_(b).add_(c * D[at])
                D[at] += P

        def over_r(name, X, inv_r, table):
            """X / r, in the PML X / r~ when the radius is stretched."""
            if not self.metric:
                return X * inv_r
            Y = X.clone()
            for n, sl in enumerate(rsl):
                key = (name, n, "m")
                if key not in psi:
                    psi[key] = [torch.zeros_like(X[sl]), _t(table[2])[sl][:, None, None], _t(table[3])[sl][:, None, None]]
                P, b, c = psi[key]
                P.mul_(b).add_(c * X[sl])
                Y[sl] += P
            return Y * inv_r

        def d_phi(F, forward):
            if self.bor:
                return 1j * s.m * F
            n = torch.roll(F, -1 if forward else 1, 1)
            if forward:
                n[:, -1] *= bloch
                return (n - F) / self.dphi
            n[:, 0] *= bloch.conjugate()
            return (F - n) / self.dphi

        def radial_curl(name, F, nb, G, inv_r, table):
            """(1/r) d(r F)/dr - (1/r) dG/dphi: all of the first term stretched, or the derivative alone."""
            sign = 1 if nb > 0 else -1
            N = _shift(F, 0, nb)
            d, mean = sign * (N - F) / s.dr, 0.5 * (N + F)
            if not self.metric:
                d = d + mean * inv_r
                stretch(name, d, 0, table)
                return d - G * inv_r
            whole = d + mean * inv_r - G * inv_r
            stretch(name, d, 0, table)
            X = mean - G
            full = d + over_r(name, X, inv_r, table)
            for sl in rsl:
                whole[sl] = full[sl]
            return whole

        mon = torch.zeros((Q, 2, s.n_r, s.n_phi), dtype=C128, device=DEV) if mon_k is not None else None
        des = torch.zeros((Q, 3, s.n_r, s.n_phi, self.nk), dtype=C128, device=DEV)
        tw = _t(self.tw, C128)
        ie_r, ie_p, ie_z = inv_eps
        dsl = slice(s.design_k0, s.design_k0 + self.nk)
        for n in range(s.n_steps):
            dz = (_shift(Ep, 2, 1) - Ep) / s.dz
            stretch("hr", dz, 2, self.cz_h)
            Hr -= dt * (over_r("hr", d_phi(Ez, True), irn, self.cr_n) - dz)
            dz = (_shift(Er, 2, 1) - Er) / s.dz
            stretch("hp", dz, 2, self.cz_h)
            dr = (_shift(Ez, 0, 1) - Ez) / s.dr
            stretch("hpr", dr, 0, self.cr_h)
            Hp -= dt * (dz - dr)
            Hz -= dt * radial_curl("hz", Ep, 1, d_phi(Er, True), irh, self.cr_h)
            del dz, dr

            dz = (Hp - _shift(Hp, 2, -1)) / s.dz
            stretch("er", dz, 2, self.cz_n)
            C = over_r("er", d_phi(Hz, False), irh, self.cr_h) - dz
            C[:, :, src_k] -= src_r(n)
            C[:, :, 0] = 0
            Er += dt * ie_r * C
            dz = (Hr - _shift(Hr, 2, -1)) / s.dz
            stretch("ep", dz, 2, self.cz_n)
            dr = (Hz - _shift(Hz, 0, -1)) / s.dr
            stretch("epr", dr, 0, self.cr_n)
            C = dz - dr
            C[:, :, src_k] -= src_p(n)
            C[:, :, 0] = 0
            C[0] = 0
            Ep += dt * ie_p * C
            C = radial_curl("ez", Hp, -1, d_phi(Hr, False), irn, self.cr_n)
            C[0] = 0
            Ez += dt * ie_z * C
            del dz, dr, C
            if mon is not None:
                mon += tw[n].view(Q, 1, 1, 1) * torch.stack([Er[:, :, mon_k], Ep[:, :, mon_k]])
            for c, F in enumerate((Er, Ep, Ez)):
                des[:, c] += tw[n].view(Q, 1, 1, 1) * F[:, :, dsl]
        return mon, des, torch.stack([Er, Ep, Ez, Hr, Hp, Hz])

    def inv_eps(self, bars):
        an, dn, ac, dc = self.eps_tables()
        return [1.0 / (a + d * b.detach()[:, :, None]) for a, d, b in ((an, dn, bars[0]), (an, dn, bars[1]), (ac, dc, bars[2]))]

    def forward(self, bars):
        s = self.s
        u = (self.n + 0.5) * self.dt - s.pulse_t0
        g = np.cos(2 * np.pi * s.pulse_f0 * u) * np.exp(-u * u / (2 * s.pulse_sigma ** 2)) * 0.5 / s.dz
        pr, pp = _t(self.ph_n, C128)[None], _t(1j * self.ph_h, C128)[None]
        return self.loop(self.inv_eps(bars), s.source_k, lambda n: g[n] * pr, lambda n: g[n] * pp, s.monitor_k)

    def focal(self, mon):
        j = np.arange(self.s.n_phi)
        z = 0 if self.bor else 1
        en, eh = (_t(np.exp(-1j * z * (j + o) * self.dphi), C128) for o in (0.0, 0.5))
        return (_t(self.Gr, C128) * (mon[:, 0] * en).sum(-1) + _t(self.Gp, C128) * (mon[:, 1] * eh).sum(-1)).sum(-1)

    def gradient(self, rho, bars, des, dI):
        """dI/drho for dI = dI/dRe S + i dI/dIm S, through the discrete adjoint run."""
        s, Q = self.s, len(self.w)
        vol = s.dr * self.dphi * s.dz
        g = (1j * np.asarray(dI.cpu()))[:, None]
        with np.errstate(divide="ignore", invalid="ignore"):
            br = g * self.Gr.conj() / (self.wt[:, None] * self.rh * vol)
            bp = np.where(self.rn > 0, g * self.Gp.conj() / (self.wt[:, None] * self.rn * vol), 0.0)

        def base(l, n):
            u = n * self.dt - 6 * s.pulse_sigma
            return np.exp(1j * self.w[l] * u - u * u / (2 * s.pulse_sigma ** 2))
        pulses = np.stack([base(l, self.n + 1) - base(l, self.n) for l in range(Q)], 1)
        spec = np.exp(-1j * self.w[None] * ((self.n + 0.5) * self.dt)[:, None]) * self.dt
        prof = pulses @ np.linalg.inv(pulses.T @ spec).T
        prof, br, bp = _t(prof, C128), _t(br, C128), _t(bp, C128)
        pr, pp = _t(self.ph_n, C128)[None], _t(self.ph_h, C128)[None]
        _, adj, _ = self.loop(self.inv_eps(bars), s.monitor_k, lambda n: (prof[n] @ br)[:, None] * pr,
                              lambda n: (prof[n] @ bp)[:, None] * pp, None)
        opp = np.r_[Q // 2:Q, 0:Q // 2]
        w2 = _t(self.wt ** 2).view(Q, 1, 1, 1, 1)
        G = (w2 * (des * adj[opp].conj()).real).sum(0)
        radius = [_t(x)[:, None, None] * vol for x in (self.rh, self.rn, self.rn)]
        tables = self.eps_tables()
        sl = slice(s.design_k0, s.design_k0 + self.nk)
        total = 0.0
        for c, d in enumerate((tables[1], tables[1], tables[3])):
            total = total + (bars[c] * (G[c] * radius[c] * d[sl]).sum(-1)).sum()
        return torch.autograd.grad(total, rho)[0]


def _net64(case, seed):
    """Layers of the network as 64-bit torch tensors [out][in][k][k] with their biases."""
    v = _t(_net_params(case, seed))
    out, o = [], 0
    for k, ci, co, _ in _layers(1, case.get("out_ch", 24)):
        n = co * k * k * ci
        out.append((v[o:o + n].view(co, k, k, ci).permute(0, 3, 1, 2).contiguous(), v[o + n:o + n + co].clone()))
        o += n + co
    return out


def _unet(layers, x):
    """x [n][1][H][W] -> [n][C][H][W]."""
    F = torch.nn.functional
    it = iter(layers)

    def conv(h, act=True):
        w, b = next(it)
        # convolution as a matrix product over shifted copies: library FP64 convolutions are slow here
        k, (n, c, H, W) = w.shape[2], h.shape
        cols = F.unfold(h, k, padding=k // 2)
        y = (w.reshape(w.shape[0], -1) @ cols).view(n, -1, H, W) + b.view(1, -1, 1, 1)
        return F.relu(y) if act else y

    skips = []
    for _ in range(3):
        x = conv(conv(x))
        skips.append(x)
        x = F.avg_pool2d(x, 2)
    x = conv(conv(x))
    for _ in range(3):
        x = conv(conv(torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"), skips.pop()], 1)))
    return conv(x, act=False)


def _chunks(case):
    per = max(1, (1 << 17) // (case["height"] * case["width"]))
    return [slice(k, min(k + per, case["batch"])) for k in range(0, case["batch"], per)]


def exact(case, seed):
    if case["kind"] == "zone":
        spec = _spec(case)
        sol = _Solver(spec, case.get("radial_pml", 0))
        rho = _rho(spec, seed).to(F64).requires_grad_(True)
        bars = sol.bars(rho)
        mon, des, fields = sol.forward(bars)
        S = sol.focal(mon)
        if case["run"] == "forward":
            return {"S": S.cpu().numpy(), "monitor": mon, "fields": fields}
        return {"I": float(2 * (S.abs() ** 2).sum()), "grad": sol.gradient(rho, bars, des, 4 * S), "monitor": mon}
    if case["kind"] == "lens":
        zones = []
        for i, spec in enumerate(_lens_specs(case)):
            sol = _Solver(spec, 0)
            rho = _rho(spec, seed + 100 * i).to(F64).requires_grad_(True)
            bars = sol.bars(rho)
            mon, des, _ = sol.forward(bars)
            zones.append((sol, rho, bars, des, sol.focal(mon)))
        S = sum(z[4] for z in zones)
        return {"S": S.cpu().numpy(), "grads": [sol.gradient(rho, bars, des, 4 * S) for sol, rho, bars, des, _ in zones]}
    if case["kind"] == "ascent":
        spec = _patch(case)
        sol = _Solver(spec, 0)
        rho = torch.tensor(smoothed_rho(spec.n_r_design, spec.n_phi, seed, mode="minmax"), dtype=torch.float32, device=DEV).to(F64).requires_grad_(True)
        y = _unet(_net64(case, seed), sol.tilde(rho)[None, None])[0] * 0.25
        y = y.view(len(sol.w), 2, 2, spec.n_r_design, spec.n_phi)
        mon = torch.nn.functional.pad(torch.complex(y[:, :, 0], y[:, :, 1]), (0, 0, sol.i0, spec.n_r - sol.i1))
        value = 2 * (sol.focal(mon).abs() ** 2).sum()
        return {"I": float(value), "grad": torch.autograd.grad(value, rho)[0]}
    layers = _net64(case, seed)
    x, target = _net_data(case, seed)
    if case["run"] == "forward":
        with torch.no_grad():
            return {"y": torch.cat([_unet(layers, x[c].to(F64).permute(0, 3, 1, 2)).permute(0, 2, 3, 1) for c in _chunks(case)])}
    for w, b in layers:
        w.requires_grad_(True)
        b.requires_grad_(True)
    flat = [t for wb in layers for t in wb]
    loss, grads = 0.0, None
    for c in _chunks(case):
        y = _unet(layers, x[c].to(F64).permute(0, 3, 1, 2)).permute(0, 2, 3, 1)
        part = ((y - target[c].to(F64)) ** 2).sum() / target.numel()
        got = torch.autograd.grad(part, flat)
        loss += float(part.detach())
        grads = got if grads is None else [a + b for a, b in zip(grads, got)]
    parts = [g.permute(0, 2, 3, 1).reshape(-1) if g.dim() == 4 else g for g in grads]
    return {"loss": torch.tensor([loss], dtype=F64), "grads": torch.cat(parts)}
