"""What the speed of this library is measured on: its work as a user's program calls it, at listed sizes and at drawn ones.

Three kinds of work, each through the public calls of the package:

  grid       a wave packet on a 2-D (x-z) or 3-D grid: dirac_set_state, a few dirac_step calls with dirac_observables after
             each (a program that follows a packet reads the norm, the centroid and the face flux as it goes), dirac_get_state.
             FP64, FP32 and fixed-point states, first- and second-order splitting, zero and periodic boundaries, a Klein step or
             a soft Coulomb well, absorbing layers, a laser field (uniform or varying in space) and characteristic shifts.
  ensemble   many independent Klein-step runs of uneven sizes and step counts: dirac_batch_reset, _run, _results.
  surrogate  the transmission network: dirac_surrogate_predict on host queries, and dirac_surrogate_train.

listed() says for each case what it stands for.  draw() spreads over the same ranges: 2-D grids from 96 to 2048 cells a side,
3-D grids from 24 to 256, 1 to a few hundred steps, ensembles of 2 to 24 runs, 1 to 200,000 queries, training batches of 64 to
1024.  exact() is the same mathematics in plain 64-bit torch."""
import math

import numpy as np
import torch

import paper_1107_4650_gb300 as D

C, M = 137.0359895, 1.0          # atomic units
DX = 10.0 / 8192.0               # the paper's 2-D mesh spacing
PRECISION = {"fp64": 0, "fp32": 1, "fx64": 2}
BOX_LO, BOX_HI = (0.5, 0.2, 40.0), (3.0, 1.0, 150.0)  # the surrogate's box: V0 / mc^2, p0 / mc, width / dx
SIDES = (256, 384, 512, 768, 1024)


def _grid(name, n, precision, steps, calls=1, splitting="lie", boundary="zero", potential="none", field="none", absorb=0,
          shift=1):
    case = {"kind": "grid", "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision, "steps": steps, "calls": calls,
            "splitting": splitting, "boundary": boundary, "potential": potential, "field": field, "absorb": absorb,
            "shift": shift}
    return dict(case, name=name) if name else case


def listed():
    return [
        # A free packet on the small grid of the accuracy studies (256 x 256, 200 steps), followed by its observables: the
        # smallest calls, where launches and latency count.
        _grid("free_256_fp64", (256, 1, 256), "fp64", 200, calls=8),
        # The Klein step at its full size, in the precision the results are quoted in: the library's headline workload.
        _grid("klein_2048_fp64", (2048, 1, 2048), "fp64", 40, potential="step"),
        # The same run with FP32 storage, as parameter scans use it.
        _grid("klein_2048_fp32", (2048, 1, 2048), "fp32", 200, potential="step"),
        # Fixed point with absorbing layers on a ragged grid (sizes that fill no tile): the fast form of an FP64-accurate run.
        _grid("klein_1531x1087_fx64", (1531, 1, 1087), "fx64", 100, potential="step", absorb=64),
        # Second-order steps in a laser pulse on a periodic ragged grid, FP64.
        _grid("laser_strang_1000x777_fp64", (1000, 1, 777), "fp64", 40, splitting="strang", boundary="periodic",
              field="laser"),
        # A small FP32 periodic box with second-order steps and many short calls: an interactive run.
        _grid("strang_301x257_fp32", (301, 1, 257), "fp32", 300, calls=6, splitting="strang", boundary="periodic",
              potential="step"),
        # A packet in a soft Coulomb well in 3-D, FP64.
        _grid("coulomb_256_fp64", (256, 256, 256), "fp64", 8, potential="coulomb"),
        # The same at the largest size in use, FP32 storage.
        _grid("coulomb_384_fp32", (384, 384, 384), "fp32", 20, potential="coulomb"),
        # Second-order 3-D steps on a ragged FP32 box.
        _grid("strang3d_200x144x177_fp32", (200, 144, 177), "fp32", 12, splitting="strang", potential="coulomb"),
        # Uneven Klein runs advanced together, as the training labels of the surrogate and scans are made.
        {"name": "ensemble_24_fp32", "kind": "ensemble", "runs": 24, "precision": "fp32"},
        # Queries of the trained network, one service call.
        {"name": "predict_4096", "kind": "predict", "n": 4096},
        # One epoch of training on 20,000 samples in the script's mini-batches.
        {"name": "train_20000", "kind": "train", "n": 20000, "batch": 256, "epochs": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid2"] * 6 + ["grid3"] * 3 + ["ensemble", "predict", "train"])
    if kind == "ensemble":
        return {"kind": "ensemble", "runs": _log(rng, 2, 16), "precision": "fp32"}
    if kind == "predict":
        return {"kind": "predict", "n": _log(rng, 1, 200000)}
    if kind == "train":
        return {"kind": "train", "n": _log(rng, 1500, 20000), "batch": _log(rng, 64, 1024), "epochs": 1}
    three = kind == "grid3"
    precision = rng.choice(["fp64", "fp64", "fp32", "fp32", "fx64"])
    splitting = rng.choice(["lie", "lie", "strang"])
    field = "none" if precision == "fx64" else rng.choice(["none", "none", "none", "laser", "cell"])
    shift = 1 if precision == "fx64" or field == "cell" else rng.choice([1, 1, 1, 1, 2, 3])
    n = [_log(rng, 24, 256) if three else _log(rng, 96, 2048) for _ in range(3)]
    if not three:
        n[1] = 1
    cells = n[0] * n[1] * n[2]
    # no more point-steps than a few tens of milliseconds of the slowest form
    most = max(1, int(1.0e8 / cells))
    steps = max(1, min(_log(rng, 4, 300), most))
    return _grid(None, n, precision, steps, calls=min(steps, rng.choice([1, 1, 2, 5])), splitting=splitting,
                 boundary=rng.choice(["zero", "zero", "periodic"]),
                 potential=rng.choice(["coulomb", "none"]) if three else rng.choice(["step", "step", "none"]), field=field,
                 absorb=rng.choice([0, 0, 0, min(32, n[0] // 4)]), shift=shift)


# ------------------------------------------------------------------------------------------------ inputs

def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _ndim(case):
    return 3 if case["ny"] > 1 else 2


def _dt(case):
    per = {"lie": 1.0, "strang": 4.0 if _ndim(case) == 3 else 2.0}[case["splitting"]]
    return per * case["shift"] * DX / C


def _face(case):
    return (5 * case["nx"]) // 8


def _centres(n):
    return (np.arange(n) + 0.5 - 0.5 * n) * DX


def _grid_inputs(case, seed):
    """psi (complex128, on the GPU, [z][y][x][4]), V (host, or None), absorber (host, or None), field (dict of host arrays)."""
    rng = np.random.default_rng([seed, 1107])
    nx, ny, nz = _dims(case)
    three = _ndim(case) == 3
    width = rng.uniform(0.05, 0.08) * min(nx, nz, ny if three else nx) * DX
    k0 = rng.uniform(0.2, 1.0) * M * C
    face_x = (_face(case) - 0.5 * nx) * DX
    x0 = face_x - 4 * width if case["potential"] == "step" else rng.uniform(-0.1, 0.1) * nx * DX
    y0 = rng.uniform(-0.1, 0.1) * ny * DX if three else 0.0
    z0 = rng.uniform(0.03, 0.1) * nz * DX
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    line = lambda n, at: np.exp(-((_centres(n) - at) ** 2) / (4 * width ** 2))  # noqa: E731
    gx = cuda(line(nx, x0) * np.exp(1j * k0 * _centres(nx)))
    gy = cuda(line(ny, y0) if three else np.ones(1))
    gz = cuda(line(nz, z0))
    spin = cuda(np.array([1.0, 0.0, 0.0, C * k0 / (M * C * C + math.sqrt(M * M * C ** 4 + C * C * k0 * k0))]))
    norm = torch.sqrt((gx.abs() ** 2).sum() * (gy ** 2).sum() * (gz ** 2).sum() * (spin ** 2).sum() * DX ** _ndim(case))
    psi = (gz[:, None, None] * gy[None, :, None]).unsqueeze(-1) * (gx[:, None] * (spin / norm))[None, None]
    V = None
    if case["potential"] == "step":
        V0 = rng.uniform(0.5, 3.0) * M * C * C
        V = 0.5 * V0 * (1.0 + np.tanh((_centres(nx) - face_x) / (4 * DX)))
    elif case["potential"] == "coulomb":
        Z = rng.uniform(1.0, 20.0)
        x2, y2, z2 = (cuda(_centres(k) ** 2) for k in (nx, ny, nz))
        V = (-Z / torch.sqrt(x2[None, None, :] + y2[None, :, None] + z2[:, None, None] + (2 * DX) ** 2)).cpu().numpy()
    absorber = None
    if case["absorb"]:
        i, w = np.arange(nx), case["absorb"]
        s = np.maximum(np.clip((w - i) / w, 0, 1), np.clip((i - (nx - w) + 1) / w, 0, 1))
        absorber = np.exp(-0.1 * s * s)
    field = {}
    if case["field"] != "none":
        # a sin^2 pulse over the run, its integral over each step by the midpoint value
        t = (np.arange(case["steps"]) + 0.5) / case["steps"]
        pulse = np.sin(np.pi * t) ** 2 * np.sin(4 * np.pi * t + rng.uniform(0, 6)) * _dt(case)
        e = rng.normal(size=3)
        A = 0.3 * C * C * pulse[:, None] * (e / np.linalg.norm(e))[None, :]
        if case["field"] == "laser":
            field["A"] = np.ascontiguousarray(A)
        else:
            phase = 2 * np.pi * (_centres(nx)[None, None, :] / (nx * DX) + 0.5 * _centres(nz)[:, None, None] / (nz * DX))
            prof = np.broadcast_to(np.cos(phase), (nz, ny, nx))
            field["a"] = np.ascontiguousarray(np.broadcast_to(prof[..., None], (nz, ny, nx, 3)))
            field["w"] = np.ascontiguousarray(np.broadcast_to(1.0 + 0.5 * np.sin(phase), (nz, ny, nx)))
            field["F"] = np.ascontiguousarray(np.concatenate([A, (0.2 * C * C * pulse)[:, None]], axis=1))
    return psi, V, absorber, field


def _runs(case, seed):
    rng = np.random.default_rng([seed, 2011])
    out = []
    for _ in range(case["runs"]):
        side = int(rng.choice(SIDES))
        V0, p0 = rng.uniform(0.5, 3.0) * M * C * C, rng.uniform(0.2, 1.0) * M * C
        w = min(rng.uniform(40, 150), (side - 8 - 32 - 32) / 8.0)  # the packet fits its side
        E = math.sqrt(p0 * p0 * C * C + M * M * C ** 4)
        nsteps = int(np.clip(math.ceil(8 * w / (p0 * C / E)) + 200, 2000, 6000))
        out.append({"side": side, "face": min(int(math.ceil(8 * w)) + 24, side - 48), "nsteps": nsteps, "V0": V0,
                    "L": 4 * DX, "p0": p0, "width": w * DX, "x0": -4 * w * DX, "absorb": 16, "eta": 0.1})
    return out


def _network(seed):
    """FP32 parameters of the 3-256-256-256-256-1 network, as a seeded initialisation gives them."""
    rng = np.random.default_rng([seed, 256])
    parts = []
    for fan_in, fan_out in ((3, 256), (256, 256), (256, 256), (256, 256), (256, 1)):
        a = math.sqrt(6.0 / (fan_in + fan_out))
        parts += [rng.uniform(-a, a, fan_in * fan_out), 0.1 * rng.uniform(-1, 1, fan_out)]
    return np.concatenate(parts).astype(np.float32)


def _queries(seed, n):
    rng = np.random.default_rng([seed, 3])
    lo, hi = np.array(BOX_LO), np.array(BOX_HI)
    return lo + (hi - lo) * rng.uniform(0.0, 1.0, (n, 3))


def _labels(X):
    """Transmissions of the size and shape the solver's have: near 0 in the gap, up to about 0.9 either side of it."""
    E = np.sqrt(1.0 + X[:, 1] ** 2)
    return 0.9 / (1.0 + np.exp(-(np.abs(X[:, 0] - E) - 1.0) * X[:, 2] / 20.0))


class _Handle:
    """A library handle that is given back when its owner drops it."""

    def __init__(self, handle, destroy):
        self.h, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.h)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "grid":
        psi, V, absorber, field = _grid_inputs(case, seed)
        f32 = case["precision"] == "fp32"
        cfg = D.make_config(_dims(case), ndim=_ndim(case), precision=PRECISION[case["precision"]],
                            boundary=D.DIRAC_BC_PERIODIC if case["boundary"] == "periodic" else D.DIRAC_BC_ZERO,
                            flux_face=_face(case), splitting=D.DIRAC_STRANG if case["splitting"] == "strang" else D.DIRAC_LIE,
                            char_shift=case["shift"])
        g = _Handle(D.dirac_create_grid(cfg), D.dirac_destroy)
        if V is not None:
            D.dirac_set_potential(g.h, V, D.DIRAC_V_FULL if V.ndim == 3 else D.DIRAC_V_X_ONLY)
        if absorber is not None:
            D.dirac_set_absorber(g.h, absorber)
        if "A" in field:
            D.dirac_set_vector_potential(g.h, field["A"])
        if "F" in field:
            D.dirac_set_field(g.h, field["a"], field["w"], field["F"])
        s["psi"] = psi.to(torch.complex64) if f32 else psi
        s["out"] = torch.empty_like(s["psi"])
        s["grid"] = g
    elif case["kind"] == "ensemble":
        cfg = D.dirac_batch_default_config()
        cfg.precision = PRECISION[case["precision"]]
        runs = _runs(case, seed)
        s["batch"] = _Handle(D.dirac_batch_create(runs, cfg), D.dirac_batch_destroy)
        s["out"] = torch.empty((runs[0]["side"], 1, runs[0]["side"], 4), dtype=torch.complex64, device="cuda")
    else:
        big = case["n"] if case["kind"] == "predict" else case["batch"]
        s["net"] = _Handle(D.dirac_surrogate_create(BOX_LO, BOX_HI, seed=7, max_batch=max(4096, big)), D.dirac_surrogate_destroy)
        s["params"] = _network(seed)
        D.dirac_surrogate_set_params(s["net"].h, s["params"])
        s["X"] = _queries(seed, case["n"])
        s["T"] = _labels(s["X"])
    return s


# ------------------------------------------------------------------------------------------------ the calls

def run(s):
    case = s["case"]
    if case["kind"] == "grid":
        h, obs, done = s["grid"].h, [], 0
        D.dirac_set_state(h, s["psi"])
        for k in range(case["calls"]):
            upto = case["steps"] * (k + 1) // case["calls"]
            D.dirac_step(h, upto - done)
            done = upto
            obs.append(D.dirac_observables(h))
        D.dirac_get_state(h, s["out"])
        return {"psi": s["out"], "observables": obs}
    if case["kind"] == "ensemble":
        h = s["batch"].h
        D.dirac_batch_reset(h)
        D.dirac_batch_run(h)
        results = D.dirac_batch_results(h, case["runs"])
        D.dirac_batch_get_state(h, 0, s["out"])  # one run's final packet, for its density map
        return dict(results, psi0=s["out"])
    if case["kind"] == "predict":
        return D.dirac_surrogate_predict(s["net"].h, s["X"])
    h = s["net"].h
    D.dirac_surrogate_set_params(h, s["params"])
    loss = D.dirac_surrogate_train(h, s["X"], s["T"], case["epochs"], case["batch"], 1e-3)
    return {"loss": loss, "params": D.dirac_surrogate_get_params(h)}


def work(case):
    if case["kind"] == "grid":
        cells = case["nx"] * case["ny"] * case["nz"]
        state = cells * (32 if case["precision"] == "fp32" else 64)
        table = (cells if case["potential"] == "coulomb" else case["nx"]) * (16 if case["precision"] == "fp32" else 32)
        sweeps = _ndim(case) if case["splitting"] == "lie" else (8 if _ndim(case) == 3 else 4)
        phase = 24 if case["field"] == "none" else 96
        # each call's state comes in and goes out once; each sweep adds 16 numbers a cell
        return {"bytes": 2.0 * state + table, "flops": float(cells) * case["steps"] * (16 * sweeps + phase)}
    if case["kind"] == "ensemble":
        runs = _runs(case, 1)  # a typical draw of the sizes
        return {"bytes": 32.0 * sum(r["side"] ** 2 for r in runs), "flops": 56.0 * sum(r["side"] ** 2 * r["nsteps"] for r in runs)}
    flops = 2.0 * (3 * 256 + 3 * 256 * 256 + 256)
    params = 3 * 256 + 3 * 256 * 256 + 256 + 4 * 256 + 1
    if case["kind"] == "predict":
        return {"bytes": 32.0 * case["n"] + 2.0 * params, "flops": flops * case["n"]}
    return {"bytes": 32.0 * case["n"] + 8.0 * params, "flops": 3 * flops * case["n"] * case["epochs"]}


# ------------------------------------------------------------------------------------------------ 64-bit values

_ALPHA = {0: np.array([[0, 0, 0, 1], [0, 0, 1, 0], [0, 1, 0, 0], [1, 0, 0, 0]], complex),
          1: np.array([[0, 0, 0, -1j], [0, 0, 1j, 0], [0, -1j, 0, 0], [1j, 0, 0, 0]], complex),
          2: np.array([[0, 0, 1, 0], [0, 0, 0, -1], [1, 0, 0, 0], [0, -1, 0, 0]], complex)}


def _moved(a, axis, by, periodic):
    """a(i - by) along a grid axis (0 x, 1 y, 2 z), zero or wrapped outside."""
    d = 2 - axis
    out = torch.roll(a, by, d)
    if not periodic:
        n = a.shape[d]
        out.narrow(d, 0 if by > 0 else max(0, n + by), min(n, abs(by))).zero_()
    return out


def _sweep(psi, axis, K, periodic, flux):
    """psi'(i) = 1/2 [(1 + alpha) psi(i - K) + (1 - alpha) psi(i + K)], and the probability that crosses the face."""
    rows = [(int(np.flatnonzero(r)[0]), complex(r[np.flatnonzero(r)[0]])) for r in _ALPHA[axis]]
    turned = torch.stack([psi[..., j] * v for j, v in rows], dim=-1)
    plus, minus = 0.5 * (psi + turned), 0.5 * (psi - turned)
    if axis == 0 and flux is not None:
        f, n = flux["face"], psi.shape[2]
        at = lambda a, i: (a[:, :, i].abs() ** 2).sum() if 0 <= i < n else 0.0  # noqa: E731
        flux["sum"] = flux["sum"] + sum(at(plus, f - 1 - j) - at(minus, f + j) for j in range(K))
    del turned
    out = _moved(plus, axis, K, periodic)
    out += _moved(minus, axis, -K, periodic)
    return out


def _phase(psi, mu, vdt, absorber, At):
    """exp(-i (beta mu - alpha . At)) exp(-i vdt), per cell where vdt or At vary, times the absorber's factors."""
    if At is None:
        sign = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=psi.device)
        for c in range(4):
            t = vdt + mu * sign[c]
            psi[..., c] *= torch.complex(torch.cos(t), -torch.sin(t)) * absorber
        return psi
    size = torch.sqrt(mu * mu + At[0] ** 2 + At[1] ** 2 + At[2] ** 2)
    cs, sn = torch.cos(size), torch.sin(size) / size
    g = torch.complex(torch.cos(vdt), -torch.sin(vdt)) * absorber
    beta = (1.0, 1.0, -1.0, -1.0)
    out = torch.empty_like(psi)
    for r in range(4):
        acc = psi[..., r] * (cs - 1j * mu * beta[r] * sn)
        for d in range(3):
            j = int(np.flatnonzero(_ALPHA[d][r])[0])
            acc = acc + psi[..., j] * (1j * complex(_ALPHA[d][r][j]) * At[d] * sn)
        out[..., r] = acc * g
    return out


def _observe(psi, case, flux, step):
    nx, ny, nz = _dims(case)
    vol = DX ** _ndim(case)
    rho = (psi.real ** 2 + psi.imag ** 2).sum(-1)
    total = rho.sum()
    x, y, z = (torch.from_numpy(_centres(k)).to(rho.device) for k in (nx, ny, nz))
    return {"norm": float(total * vol), "norm_right": float(rho[:, :, _face(case):].sum() * vol),
            "flux_cum": float(flux["sum"] * vol),
            "centroid": tuple(float(v / total) for v in ((rho.sum((0, 1)) * x).sum(), (rho.sum((0, 2)) * y).sum(),
                                                         (rho.sum((1, 2)) * z).sum())), "step": step}


def _exact_grid(case, seed):
    psi, V, absorber, field = _grid_inputs(case, seed)
    if case["precision"] == "fp32":
        psi = psi.to(torch.complex64).to(torch.complex128)  # the values the call is given
    dev, per, K, three = psi.device, case["boundary"] == "periodic", case["shift"], _ndim(case) == 3
    cuda = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
    dt = _dt(case)
    mu = M * C * C * dt
    vdt0 = cuda(V * dt) if V is not None else torch.zeros(1, dtype=torch.float64, device=dev)
    damp = cuda(absorber) if absorber is not None else 1.0
    if case["splitting"] == "lie":
        half = [(0, K), (1, K), (2, K)] if three else [(0, K), (2, K)]
    else:
        half = [(0, K), (1, 2 * K), (0, K), (2, 2 * K)] if three else [(0, K), (2, K)]
    a, w = (cuda(field[k]) if k in field else None for k in ("a", "w"))
    flux = {"face": _face(case), "sum": torch.zeros((), dtype=torch.float64, device=dev)}
    obs, done = [], 0
    for k in range(case["calls"]):
        upto = case["steps"] * (k + 1) // case["calls"]
        for n in range(done, upto):
            for axis, by in half:
                psi = _sweep(psi, axis, by, per, flux)
            At, vdt = None, vdt0
            if "A" in field:
                At = [torch.tensor(float(v), dtype=torch.float64, device=dev) for v in field["A"][n]]
            elif "F" in field:
                At = [a[..., d] * float(field["F"][n, d]) for d in range(3)]
                vdt = vdt0 + w * float(field["F"][n, 3])
            psi = _phase(psi, mu, vdt, damp, At)
            if case["splitting"] == "strang":
                for axis, by in reversed(half):
                    psi = _sweep(psi, axis, by, per, flux)
        done = upto
        obs.append(_observe(psi, case, flux, done))
    return {"psi": psi, "observables": obs}


def _unit(seed, i):
    """Uniform numbers in [0, 1) from a splitmix64 stream."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) * np.uint64(0x100000001B3) + np.asarray(i, dtype=np.uint64) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _unpack(p):
    out, o = [], 0
    for fan_in, fan_out in ((3, 256), (256, 256), (256, 256), (256, 256), (256, 1)):
        out.append((p[o:o + fan_in * fan_out].view(fan_out, fan_in), p[o + fan_in * fan_out:o + (fan_in + 1) * fan_out]))
        o += (fan_in + 1) * fan_out
    return out


def _net(p, x):
    layers = _unpack(p)
    for W, b in layers[:-1]:
        x = torch.tanh(x @ W.T + b)
    return torch.sigmoid(x @ layers[-1][0].T + layers[-1][1])[:, 0]


def _inputs01(X):
    lo, hi = np.array(BOX_LO), np.array(BOX_HI)
    return torch.from_numpy(2.0 * (X - lo) / (hi - lo) - 1.0).cuda()


def _exact_train(case, seed):
    X = _queries(seed, case["n"])
    x, t = _inputs01(X), torch.from_numpy(_labels(X)).cuda()
    p = torch.from_numpy(_network(seed).astype(np.float64)).cuda()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    n, per = case["n"], max(1, case["n"] // case["batch"])
    size = case["batch"] if case["n"] >= case["batch"] else case["n"]
    step, loss = 0, 0.0
    for ep in range(case["epochs"]):
        u = _unit(7 ^ 0xA5A5A5A5, ep * n + np.arange(n))
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            j = min(int(u[i] * (i + 1)), i)
            perm[i], perm[j] = perm[j], perm[i]
        perm, loss = torch.tensor(perm, device=x.device), 0.0
        for b in range(per):
            idx = perm[b * size:(b + 1) * size]
            q = p.detach().requires_grad_(True)
            err = ((_net(q, x[idx]) - t[idx]) ** 2).mean()
            (grad,) = torch.autograd.grad(err, q)
            lr = 1e-3 / 20 + 0.5 * (1e-3 - 1e-3 / 20) * (1 + math.cos(math.pi * step / (per * case["epochs"])))
            step += 1
            m, v = 0.9 * m + 0.1 * grad, 0.999 * v + 0.001 * grad * grad
            p = p - lr * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
            loss += float(err.detach()) / per
    return {"loss": loss, "params": p}


def exact(case, seed):
    if case["kind"] == "grid":
        return _exact_grid(case, seed)
    if case["kind"] == "ensemble":
        return None  # thousands of steps of each of many runs: minutes in plain torch
    if case["kind"] == "predict":
        p = torch.from_numpy(_network(seed).astype(np.float64)).cuda()
        return _net(p, _inputs01(_queries(seed, case["n"])))
    return _exact_train(case, seed)
