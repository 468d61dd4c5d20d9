"""The work that is measured: filling runs of single lattices, batched sweeps and the l(t) surrogate.

Every case goes through the package's public entry points (Lattice, Batch, MLP) as a program of a
user calls them.  Three families:

  lattice   a filling run: the initial fields go in, the lattice advances `steps` time steps with the
            FP64 reductions (l, l_vol, mass, phi_sum) read every `every` steps, and the macroscopic
            fields come back to the host.  The lattice itself (geometry, parameters, device memory and,
            with `tune`, its autotuned tile) is what a program keeps between runs.
  sweep     a batch of uneven capillaries in one persistent launch, with l(t) sampled on the way.
  mlp       the surrogate network: training from given weights, one gradient, predictions.

Bytes of work(): the stored state is read once and written once per time step (the bytes per node
update of the storage; solid nodes excluded), plus what goes in and comes out; for the network, the
rows, the targets, the results and one reading of the weights per pass over the data.
"""
import math

import numpy as np
import torch

import workloads as W
from paper_0911_0459_gb300 import (STORAGE_F16_BLOCKED, STORAGE_F32, STORAGE_F32_BLOCKED, STORAGE_F64,
                                   STORAGE_MOMENTS, Batch, Lattice)
from paper_0911_0459_gb300.lb import STORAGE_F16DEV, STORAGE_F32_GELIM, STORAGE_MOMENTS_F16
from paper_0911_0459_gb300.mlp import MLP

STORAGES = {"f64": STORAGE_F64, "f32": STORAGE_F32, "f32b": STORAGE_F32_BLOCKED, "f16dev": STORAGE_F16DEV,
            "f16b": STORAGE_F16_BLOCKED, "moments": STORAGE_MOMENTS, "moments_f16": STORAGE_MOMENTS_F16,
            "gelim": STORAGE_F32_GELIM}
# bytes read and written per node update
UPDATE_BYTES = {"f64": 288, "f32": 144, "f32b": 144, "f16dev": 76, "f16b": 76, "moments": 48, "moments_f16": 28,
                "gelim": 80}
LG_FLOPS, BINARY_FLOPS = 159, 230  # per node update: the pair-form collision, stencils and row sums


def _lattice(name, model, storage, nx, ny, x0, length, y0, h, gas, steps, every, nu_l, nu_g, theta, tune=False,
             lut=0):
    return {"name": name, "kind": "lattice", "model": model, "storage": storage, "nx": nx, "ny": ny, "x0": x0,
            "len": length, "y0": y0, "h": h, "gas": gas, "l0": 10, "steps": steps, "every": every, "nu_l": nu_l,
            "nu_g": nu_g, "theta": theta, "tune": tune, "nu_table": lut}


def listed():
    return [
        # the liquid-gas capillary of the command line, FP64, l(t) every 50 steps: the smallest lattice, latency
        _lattice("lg_256x32_f64", "lg", "f64", 256, 32, 64, 192, 4, 24, 16, 400, 50, 1 / 6, 1 / 6, 60.0),
        # the paper's own 700 x 40 layout (rows that are no multiple of 8 nodes), the command line's default
        # storage and output interval, default kernel and tile
        _lattice("paper_700x40_f32", "binary", "f32", 700, 40, 350, 350, 0, 39, 16, 1000, 100, 1.17, 0.017, 60.0),
        # the Washburn run of the command line: a lattice that stays in L2, FP32 planes, default tile
        _lattice("binary_2048x64_f32", "binary", "f32", 2048, 64, 256, 1792, 7, 50, 64, 1000, 100, 0.83, 0.083, 60.0),
        # the crop the precision report runs, FP32 blocks, autotuned as in the usage example
        _lattice("crop_1024x64_f32b", "binary", "f32b", 1024, 64, 256, 768, 7, 50, 64, 2000, 500, 0.83, 0.0166, 45.0,
                 True),
        # the large capillary of the benchmark in its FP32 blocks, autotuned
        _lattice("large_16384x256_f32b", "binary", "f32b", 16384, 256, 512, 15872, 28, 200, 128, 1000, 100, 0.83,
                 0.0166, 45.0, True),
        # the same in FP16 deviations, default tile
        _lattice("large_16384x256_f16b", "binary", "f16b", 16384, 256, 512, 15872, 28, 200, 128, 1000, 100, 0.83,
                 0.0166, 45.0),
        # the same in six moments, autotuned
        _lattice("large_16384x256_moments", "binary", "moments", 16384, 256, 512, 15872, 28, 200, 128, 1000, 100,
                 0.83, 0.0166, 45.0, True),
        # the liquid-gas model in FP64 on the large capillary
        _lattice("lg_16384x256_f64", "lg", "f64", 16384, 256, 512, 15872, 28, 200, 128, 100, 50, 1 / 6, 1 / 6, 60.0),
        # the sweep of 256 uneven capillaries, in the storage the surrogate's data are made with
        {"name": "sweep_256_f32b", "kind": "sweep", "storage": "f32b", "n": 256, "sizes": 0, "fixed_len": 0,
         "steps": 80, "samples": 4, "align": 8},
        # training the surrogate: 4096 curves, five members, from given weights
        {"name": "mlp_train_4096", "kind": "mlp", "what": "train", "n_in": 4, "hidden": 256, "n_out": 64,
         "members": 5, "rows": 4096, "steps": 100},
        # one query batch of the surrogate: the smallest call, latency
        {"name": "mlp_predict_512", "kind": "mlp", "what": "predict", "n_in": 4, "hidden": 256, "n_out": 64,
         "members": 5, "rows": 512, "steps": 1},
        # a parameter study answered by the surrogate in one call
        {"name": "mlp_predict_65536", "kind": "mlp", "what": "predict", "n_in": 4, "hidden": 256, "n_out": 64,
         "members": 5, "rows": 65536, "steps": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the listed ranges: any lattice, storage and size up to the large capillary, any sweep
    up to 256 capillaries, any network and batch around the surrogate's."""
    kind = rng.choice(["lattice", "lattice", "lattice", "sweep", "mlp", "mlp"])
    if kind == "lattice":
        model = rng.choice(["binary", "binary", "binary", "lg"])
        storage = rng.choice(["f64", "f32"]) if model == "lg" else rng.choice(sorted(STORAGES))
        nx = _log_int(rng, 200, 16384)
        if rng.random() < 0.5:
            nx -= nx % 8
        ny = _log_int(rng, 24, 256)
        h = max(8, int(ny * rng.uniform(0.6, 0.97)))
        x0 = max(48, nx // rng.choice([4, 8, 32]))
        length = nx - x0 if rng.random() < 0.7 else max(64, (nx - x0) // 2)
        ratio = rng.choice([1, 5, 10, 50])
        cost = 9.0 if storage == "f64" else 1.0  # FP64 arithmetic is scarce on this GPU
        # (in FP16 the velocities that viscosity has worn down sink into the rounding: shorter runs)
        steps = int(max(40, min(200 if "f16" in storage else 1000, 1.5e9 / (nx * ny * cost))))
        nu_l, nu_g = (1 / 6, 1 / 6) if model == "lg" else (0.83, 0.83 / ratio)
        case = _lattice("", model, storage, nx, ny, x0, length, (ny - h) // 2, h, max(8, x0 // 4), steps,
                        max(20, steps // 10), nu_l, nu_g, rng.choice([45.0, 60.0, 75.0]), rng.random() < 0.3,
                        10000 if model == "binary" and rng.random() < 0.1 else 0)
    elif kind == "sweep":
        storage = rng.choice(["f32", "f32b", "f16b", "f16dev", "moments", "moments", "f64"])
        n = _log_int(rng, 2, 256 if storage != "f64" else 24)
        case = {"kind": "sweep", "storage": storage, "n": n, "sizes": rng.randint(1, 99),
                "fixed_len": rng.choice([0, 0, 1024]), "steps": rng.randint(20, 80), "samples": rng.randint(1, 6),
                "align": rng.choice([1, 8, 8])}
    else:
        what = rng.choice(["train", "gradients", "predict", "predict"])
        case = {"kind": "mlp", "what": what, "n_in": rng.randint(1, 16), "hidden": 64 * rng.randint(1, 8),
                "n_out": 8 * rng.randint(1, 32), "members": rng.randint(1, 8),
                "rows": _log_int(rng, 16, 65536 if what == "predict" else 8192),
                "steps": rng.randint(10, 40) if what == "train" else 1}
    case.pop("name", None)
    return case


# ------------------------------------------------------------------------------------------- inputs

def _wall_grad(case):
    # the paper's liquid-gas gradient for 60 degrees, scaled by cos(theta); binary: Cahn's wall energy
    if case["model"] == "lg":
        return -0.288 * math.cos(math.radians(case["theta"]))
    c, lo, hi = math.cos(math.radians(case["theta"])), -1.0, 1.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 0.5 * ((1 + mid) ** 1.5 - (1 - mid) ** 1.5) < c else (lo, mid)
    return -lo * math.sqrt(0.5)  # A = kappa


def _solid(case):
    y, x = np.arange(case["ny"]), np.arange(case["nx"])
    tube = ((x - case["x0"]) % case["nx"]) < case["len"]
    band = ((y - case["y0"]) % case["ny"]) < case["h"]
    return (~band)[:, None] & tube[None, :]


def _fields(case, seed):
    """Initial fields: the two phases with the meniscus near the inlet, and small smooth disturbances."""
    rng = np.random.default_rng([seed, case["nx"], case["ny"]])
    nx, ny = case["nx"], case["ny"]
    x, y = np.arange(nx, dtype=np.float64), np.arange(ny, dtype=np.float64)

    def smooth(modes=3):
        out = np.zeros((ny, nx))
        for _ in range(modes):
            kx, ky = rng.integers(1, max(2, nx // 24)), rng.integers(1, max(2, ny // 12))
            a, b = rng.uniform(0, 2 * np.pi, 2)
            out += np.outer(np.cos(2 * np.pi * ky * y / ny + a), np.cos(2 * np.pi * kx * x / nx + b))
        return out / modes

    wide = 2.0 if case["model"] == "lg" else math.sqrt(2.0)
    xa, xb = float(case["gas"]), case["x0"] + case["l0"] + rng.uniform(-2, 2)
    chi = 0.5 * (np.tanh((x - xa) / wide) - np.tanh((x - xb) / wide))[None, :] * np.ones((ny, 1))
    ux, uy = 5e-3 * smooth(), 5e-3 * smooth()
    if case["model"] == "lg":
        rho, phi = (2.59 + 1.95 * chi) * (1 + 1e-3 * smooth()), None
    else:
        rho, phi = 1 + 1e-3 * smooth(), 2 * chi - 1
    return rho, ux, uy, phi


def _sweep(case, seed):
    """The sweep's sizes belong to the case; the contact angles come from the seed."""
    caps = W.sweep(seed=case["sizes"], n=case["n"], steps=case["steps"], fixed_len=case["fixed_len"] or None,
                   vary_gamma=bool(case["fixed_len"]), liquid_cols=384 if case["fixed_len"] else 128,
                   align=case["align"])
    rng = np.random.default_rng([seed, case["n"]])
    for c in caps:
        c.theta_deg = float(rng.uniform(30.0, 80.0))
    return caps


def _sweep_at(case):
    n = case["samples"]
    return [max(1, round(case["steps"] * (k + 1) / n)) for k in range(n)]


def _mlp_inputs(case, seed):
    """Normalised features, smooth curves as targets (a small scatter on top), Glorot-sized weights."""
    rng = np.random.default_rng([seed, case["rows"], case["hidden"]])
    ni, nh, no, n = case["n_in"], case["hidden"], case["n_out"], case["rows"]
    x = rng.uniform(-1.5, 1.5, (n, ni)).astype(np.float32)
    y = None
    if case["what"] != "predict":
        a, t = rng.normal(size=(ni, 3)) / math.sqrt(ni), np.linspace(0, 1, no)
        z = x @ a
        y = np.tanh(z[:, :1] + 0.5 * z[:, 1:2] * t) + 0.3 * z[:, 2:] * t * t + 0.01 * rng.normal(size=(n, no))
        y = y.astype(np.float32)
    params = []
    for _ in range(case["members"]):
        w = [rng.uniform(-1, 1, (o, i)) * math.sqrt(6 / (o + i)) for o, i in ((nh, ni), (nh, nh), (no, nh))]
        b = [0.05 * rng.normal(size=o) for o in (nh, nh, no)]
        params.append(np.concatenate([v.ravel() for p in zip(w, b) for v in p]).astype(np.float32))
    return x, y, params


# ---------------------------------------------------------------------------------------- the calls

def prepare(case, seed):
    if case["kind"] == "lattice":
        lg = case["model"] == "lg"
        lat = Lattice(case["nx"], case["ny"], model=0 if lg else 1, storage=STORAGES[case["storage"]],
                      tube_x0=case["x0"], tube_len=case["len"], tube_y0=case["y0"], tube_h=case["h"],
                      gas_cols=case["gas"], wall_grad=_wall_grad(case), kappa=0.02 if lg else 0.04,
                      nu_l=case["nu_l"], nu_g=case["nu_g"], nu=case["nu_l"], l0=case["l0"],
                      rho_l=4.54 if lg else 1.0, rho_g=2.59 if lg else 1.0, nu_table=case["nu_table"])
        if case["tune"]:
            lat.autotune()
        return case, lat, _fields(case, seed)
    if case["kind"] == "sweep":
        batch = Batch(_sweep(case, seed), storage=STORAGES[case["storage"]])
        batch.set_tile(128, 16)
        return case, batch, _sweep_at(case)
    x, y, params = _mlp_inputs(case, seed)
    net = MLP(case["n_in"], case["hidden"], case["n_out"], members=case["members"], max_batch=case["rows"], seed=1)
    for k, p in enumerate(params):
        net.set_params(k, p)
    return case, net, (x, y, params)


def run(state):
    case, it, inputs = state
    if case["kind"] == "lattice":
        rho, ux, uy, phi = inputs
        it.init_fields(rho, ux, uy, phi)
        curve, done = [], 0
        while done < case["steps"]:
            n = min(case["every"], case["steps"] - done)
            it.step(n)
            done += n
            d = it.filled_length()
            curve.append([d["l"], d["l_vol"], d["mass"], d["phi_sum"]])
        return {"curve": np.array(curve), "fields": it.fields()}
    if case["kind"] == "sweep":
        # the state of two of the capillaries comes back with the curves
        return {"curves": it.run_sampled(inputs), "moments": [it.moments(0), it.moments(it.n - 1)]}
    x, y, params = inputs
    if case["what"] == "predict":
        return it.predict(x)
    it.set_data(x, y)
    if case["what"] == "gradients":
        got = [it.gradients(k) for k in range(it.members)]
        return {"losses": np.array([v for v, _ in got], dtype=np.float32), "gradients": [g for _, g in got]}
    for k, p in enumerate(params):  # training starts from the same weights every time
        it.set_params(k, p)
    losses = it.train(case["steps"])
    return {"losses": losses, "params": [it.get_params(k) for k in range(it.members)]}


def work(case):
    if case["kind"] == "lattice":
        fluid = case["nx"] * case["ny"] - case["len"] * (case["ny"] - case["h"])
        lg = case["model"] == "lg"
        per = UPDATE_BYTES[case["storage"]] // (2 if lg else 1)
        return {"bytes": case["steps"] * fluid * per + 64 * case["nx"] * case["ny"],
                "flops": case["steps"] * fluid * (LG_FLOPS if lg else BINARY_FLOPS)}
    if case["kind"] == "sweep":
        caps = _sweep(case, 0)
        fluid = sum(c.nx * c.ny - c.tube_len * (c.ny - c.tube_h) for c in caps)
        return {"bytes": case["steps"] * fluid * UPDATE_BYTES[case["storage"]],
                "flops": case["steps"] * fluid * BINARY_FLOPS}
    ni, nh, no, n, k = (case[v] for v in ("n_in", "hidden", "n_out", "rows", "members"))
    weights = nh * ni + nh + nh * nh + nh + no * nh + no
    macs = nh * ni + nh * nh + no * nh
    passes = {"predict": 1, "gradients": k, "train": case["steps"]}[case["what"]]
    if case["what"] == "predict":
        return {"bytes": 4 * n * (ni + 2 * no) + 4 * k * weights, "flops": 2 * macs * n * k}
    return {"bytes": passes * (4 * n * (ni + no) + (28 if case["what"] == "train" else 8) * k * weights),
            "flops": passes * 2 * (3 * macs - nh * ni) * n * k}


# ----------------------------------------------------------------------------- the same in 64 bits

E = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (-1, 1), (1, -1)]
OPP = [0, 2, 1, 4, 3, 6, 5, 8, 7]


class _Exact:
    """The scheme on whole arrays in FP64: one capillary, plain torch."""

    def __init__(self, lg, nx, ny, x0, length, y0, h, grad, kappa, A, M, nu_l, nu_g, nu, lut):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.lg, self.geo, self.grad, self.par, self.dev = lg, (nx, ny, x0, length, y0, h), grad, (kappa, A, M, nu_l,
                                                                                                   nu_g, nu, lut), dev
        s = torch.as_tensor(_solid({"nx": nx, "ny": ny, "x0": x0, "len": length, "y0": y0, "h": h}), device=dev)
        self.solid = s
        self.ns = [[self._nb(s, i - 1, j - 1) for i in range(3)] for j in range(3)]
        b = torch.zeros_like(s)
        for row in self.ns:
            for v in row:
                b = b | v
        self.bnd, self.wall = b & ~s, bool(s.any())

    @staticmethod
    def _nb(a, dx, dy):
        return torch.roll(a, (-dy, -dx), (-2, -1)) if dx or dy else a

    def _grads(self, a, grad):
        v = [[self._nb(a, i - 1, j - 1) for i in range(3)] for j in range(3)]
        if self.wall:
            g, s = [r[:] for r in v], self.ns
            for i in (0, 2):
                g[1][i] = torch.where(s[1][i], v[1][2 - i], v[1][i])
                g[i][1] = torch.where(s[i][1], v[2 - i][1] - 2 * grad, v[i][1])
                for j in (0, 2):
                    ghost = torch.where(s[2 - j][i], v[j][2 - i], v[2 - j][i] - 2 * grad)
                    g[j][i] = torch.where(s[j][i], ghost, v[j][i])
            v = g
        dx = (v[0][2] - v[0][0] + 4 * (v[1][2] - v[1][0]) + v[2][2] - v[2][0]) / 12
        dy = (v[2][0] + 4 * v[2][1] + v[2][2] - v[0][0] - 4 * v[0][1] - v[0][2]) / 12
        lap = (v[0][0] + v[0][2] + v[2][0] + v[2][2] + 4 * (v[0][1] + v[1][0] + v[1][2] + v[2][1]) - 20 * a) / 6
        return dx, dy, lap

    def _eq(self, rho, ux, uy, phi):
        kappa, A, M, nu_l, nu_g, nu, lut = self.par
        rx, ry, rlap = self._grads(rho, self.grad if self.lg else 0.0)
        ge = None
        if self.lg:
            gx, gy = rx, ry
            P0 = rho * 0.56 / (1 - rho * (2 / 21)) - 9 / 49 * rho * rho - kappa * rho * rlap
        else:
            gx, gy, plap = self._grads(phi, self.grad)
            p2 = phi * phi
            P0 = rho / 3 + A * (0.75 * p2 * p2 - 0.5 * p2) - kappa * phi * plap
            c = ((phi + 1) / 2).clamp(0, 1)
            if lut:
                c = torch.round(c * (lut - 1)) / (lut - 1)
            nu = nu_g + c * (nu_l - nu_g)
            Q = 2 * M * (A * (p2 * phi - phi) - kappa * plap)
            u3 = (ux * ux + uy * uy) / 3
            ge = [None] * 9
            for i, (ex, ey) in enumerate(E[1:], 1):
                eu = ex * ux + ey * uy
                ge[i] = (Q + phi * eu + 1.5 * phi * (eu * eu - u3)) / (3 if i < 5 else 12)
            ge[0] = phi - sum(ge[1:])
        d = ux * rx + uy * ry
        Txx, Tyy = rho * ux * ux + nu * (2 * ux * rx + d), rho * uy * uy + nu * (2 * uy * ry + d)
        Txy = rho * ux * uy + nu * (ux * ry + uy * rx)
        Gxx, Gyy, Gxy = kappa * gx * gx, kappa * gy * gy, kappa * gx * gy
        fe = [None] * 9
        for i, (ex, ey) in enumerate(E[1:], 1):
            t = Txx * ex * ex + Tyy * ey * ey + 2 * Txy * ex * ey - (Txx + Tyy) / 3
            k = (Gxx / 3 - Gyy / 6 if i < 3 else Gyy / 3 - Gxx / 6) if i < 5 else Gxy * ex * ey / 4 - (Gxx + Gyy) / 24
            fe[i] = (P0 + rho * (ex * ux + ey * uy) + 1.5 * t) / (3 if i < 5 else 12) + k
        fe[0] = rho - sum(fe[1:])
        return fe, ge, nu

    def start(self, rho, ux, uy, phi):
        put = lambda a: None if a is None else torch.as_tensor(a, dtype=torch.float64, device=self.dev)  # noqa: E731
        rho, ux, uy, phi = put(rho), put(ux), put(uy), put(phi)
        rho = torch.where(self.solid, torch.ones_like(rho), rho)
        self.f, self.g, _ = self._eq(rho, ux, uy, phi)

    def _rested(self):
        f = self.f
        jx = f[1] - f[2] + f[5] - f[6] - f[7] + f[8]
        jy = f[3] - f[4] + f[5] - f[6] + f[7] - f[8]
        return torch.where(self.bnd, 0 * jx, jx), torch.where(self.bnd, 0 * jy, jy), jx, jy

    def step(self):
        rho = sum(self.f)
        rho = torch.where(self.solid, torch.ones_like(rho), rho)
        phi = None if self.lg else sum(self.g)
        jx, jy, rx, ry = self._rested()
        fe, ge, nu = self._eq(rho, jx / rho, jy / rho, phi)
        omega = 2 / (6 * nu + 1)
        f = [v - ((ex * (rx - jx) + ey * (ry - jy)) / (3 if i < 5 else 12) if i else 0)
             for i, ((ex, ey), v) in enumerate(zip(E, self.f))]
        dev = [a - b for a, b in zip(f, fe)]
        xx = (1 - omega) / 4 * (dev[1] + dev[2] - dev[3] - dev[4])
        xy = (1 - omega) / 4 * (dev[5] + dev[6] - dev[7] - dev[8])
        for i in range(1, 9):
            fe[i] = fe[i] + (xx if i < 3 else -xx if i < 5 else xy if i < 7 else -xy)
        self.f = self._stream(fe)
        if not self.lg:
            self.g = self._stream(ge)

    def _stream(self, f):
        out = []
        for i, (ex, ey) in enumerate(E):
            v = self._nb(f[i], -ex, -ey)
            if self.wall and i:
                v = torch.where(self.ns[1 - ey][1 - ex], f[OPP[i]], v)
            out.append(v)
        return out

    def lengths(self, rho_l, rho_g):
        nx, ny, x0, L, y0, h = self.geo
        rho = self._fluid(sum(self.f))
        phi = 0 * rho if self.lg else self._fluid(sum(self.g))
        cols = (torch.arange(L, device=self.dev) + x0) % nx
        rows = (torch.arange(h, device=self.dev) + y0) % ny
        v = rho - (rho_l + rho_g) / 2 if self.lg else phi
        mid = 0.5 * (v[rows[(h - 1) // 2], cols] + v[rows[h // 2], cols]).cpu().numpy()
        hit = np.nonzero((mid[:-1] > 0) & ~(mid[1:] > 0))[0]
        if not mid[0] > 0:
            length = 0.0
        else:
            length = float(L) if not len(hit) else hit[0] + mid[hit[0]] / (mid[hit[0]] - mid[hit[0] + 1])
        q = (rho - rho_g) / (rho_l - rho_g) if self.lg else (phi + 1) / 2
        vol = float(q[rows][:, cols].sum()) / h
        return [float(length), vol, float(rho.sum()), float(phi.sum())]

    def _fluid(self, v):
        return torch.where(self.solid, torch.zeros_like(v), v)  # what a solid node holds has no meaning

    def fields(self):
        rho = sum(self.f)
        jx, jy, _, _ = self._rested()
        out = [rho, jx / rho, jy / rho, None if self.lg else sum(self.g)]
        return [None if v is None else self._fluid(v).cpu().numpy() for v in out]

    def moments(self):
        f = self.f
        _, _, jx, jy = self._rested()
        m = [sum(f), jx, jy, f[1] + f[2] - f[3] - f[4], f[5] + f[6] - f[7] - f[8], sum(self.g)]
        return torch.stack([self._fluid(v) for v in m]).cpu().numpy()


def _net(p, x, ni, nh, no):
    out, at = [], 0
    for o, i in ((nh, ni), (nh, nh), (no, nh)):
        out += [p[at:at + o * i].reshape(o, i), p[at + o * i:at + o * i + o]]
        at += o * i + o
    w1, b1, w2, b2, w3, b3 = out
    return torch.tanh(torch.tanh(x @ w1.T + b1) @ w2.T + b2) @ w3.T + b3


def exact(case, seed):
    if case["kind"] == "lattice":
        lg = case["model"] == "lg"
        ref = _Exact(lg, case["nx"], case["ny"], case["x0"], case["len"], case["y0"], case["h"], _wall_grad(case),
                     0.02 if lg else 0.04, 0.04, 0.1, case["nu_l"], case["nu_g"], case["nu_l"], case["nu_table"])
        ref.start(*_fields(case, seed))
        curve, done = [], 0
        while done < case["steps"]:
            for _ in range(min(case["every"], case["steps"] - done)):
                ref.step()
                done += 1
            curve.append(ref.lengths(4.54 if lg else 1.0, 2.59 if lg else 1.0))
        return {"curve": np.array(curve), "fields": ref.fields()}
    if case["kind"] == "sweep":
        if case["n"] * case["steps"] > 3000:  # one capillary after the other: too long
            return None
        curves, moments = [], []
        for i, c in enumerate(_sweep(case, seed)):
            p = c.params
            ref = _Exact(False, c.nx, c.ny, c.tube_x0, c.tube_len, c.tube_y0, c.tube_h, c.wall_gradient(), p.kappa,
                         p.A, p.M, p.nu_l, p.nu_g, p.nu, 0)
            x = np.arange(c.nx, dtype=np.float64)
            s = math.sqrt(2.0)
            phi = np.tanh((x - c.gas_cols) / s) - np.tanh((x - c.tube_x0 - c.l0) / s) - 1
            one = np.ones((c.ny, c.nx))
            ref.start(one, 0 * one, 0 * one, phi[None, :] * one)
            got, done = [], 0
            for at in _sweep_at(case):
                for _ in range(at - done):
                    ref.step()
                done = at
                got.append(ref.lengths(1.0, 1.0))
            curves.append(got)
            if i in (0, case["n"] - 1):
                moments.append(ref.moments())
        return {"curves": np.array(curves), "moments": moments if case["n"] > 1 else moments * 2}
    x, y, params = _mlp_inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    sizes = case["n_in"], case["hidden"], case["n_out"]
    x = torch.as_tensor(x, dtype=torch.float64, device=dev)
    y = None if y is None else torch.as_tensor(y, dtype=torch.float64, device=dev)
    params = [torch.as_tensor(p, dtype=torch.float64, device=dev) for p in params]
    if case["what"] == "predict":
        out = torch.stack([_net(p, x, *sizes) for p in params])
        sd = out.std(0) if len(params) > 1 else torch.zeros_like(out[0])
        return out.mean(0).cpu().numpy(), sd.cpu().numpy()
    if case["what"] == "gradients":
        losses, grads = [], []
        for p in params:
            p.requires_grad_(True)
            loss = ((_net(p, x, *sizes) - y) ** 2).mean()
            losses.append(float(loss))
            grads.append(torch.autograd.grad(loss, p)[0].cpu().numpy())
        return {"losses": np.array(losses), "gradients": grads}
    # training amplifies the rounding of the first gradients without bound: no 64-bit value for its end
    return None
