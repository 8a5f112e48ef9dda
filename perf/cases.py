"""Performance cases: the work a user of the library has it do, through its public calls.

Kinds of case (each a dict of plain values; `listed` gives the fixed ones, `draw` others of the
same ranges):

* ``steps``       a single grid advanced by k time steps, then a snapshot of rho, u, B
* ``closure``     the same with the learned subgrid correction attached
* ``ensemble``    many grids advanced together, then a snapshot of every member
* ``job``         a whole run: handle from page-locked host fields, steps, snapshot to the host
* ``checkpoint``  the LES-vs-DNS analysis of one state: moments, box filter, spectra, diagnostics
* ``apriori``     training pair of a fine state and the network's prediction for it
* ``gradient``    loss and parameter gradient of the network on a batch of snapshots

Snapshots are kept in the precision of the run's storage (binary16 forms: half), as a program
that writes them out does.  `exact` restates the methods in plain binary64 torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1705_09807_gb300 import lbmhd

PRECISION = {"fp64": lbmhd.LBMHD_FP64, "fp32": lbmhd.LBMHD_FP32, "fp16": lbmhd.LBMHD_FP16,
             "fp16rel": lbmhd.LBMHD_FP16_REL}
ELEM = {"fp64": 8, "fp32": 4, "fp16": 2, "fp16rel": 2}
PLANES = {"fp64": 27, "fp32": 27, "fp16": 27, "fp16rel": 29}
SNAPSHOT = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "fp16rel": torch.float16}
FLOPS_STEP = 250      # floating-point operations of one cell update
FLOPS_NET = 27648     # of one cell through the 12 -> 32 -> 32 -> 4 network
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: the 64^2 parity configuration in binary64, read out after every step
        # (a program coupled to the solver step by step): latency and launches
        dict(name="les64_fp64_single_step", kind="steps", nx=64, ny=64, steps=1, precision="fp64", delta=2.0,
             stencil=0, mrt=False, nu=5e-3),
        # an ordinary coarse LES on a ragged grid, unequal rates, nine-point gradients
        dict(name="les250x190_fp32_mrt_iso", kind="steps", nx=250, ny=190, steps=64, precision="fp32", delta=2.0,
             stencil=1, mrt=True, nu=5e-3),
        # the DNS of the paper's comparison, in binary32
        dict(name="dns2048_fp32", kind="steps", nx=2048, ny=2048, steps=16, precision="fp32", delta=0.0,
             stencil=0, mrt=False, nu=2e-3),
        # the paper's LES grid in binary64, the reference every other form is judged by
        dict(name="les1024_fp64", kind="steps", nx=1024, ny=1024, steps=8, precision="fp64", delta=2.0,
             stencil=0, mrt=False, nu=4e-3),
        # the precision study's grid in binary16 storage
        dict(name="les4096_fp16", kind="steps", nx=4096, ny=4096, steps=8, precision="fp16", delta=2.0,
             stencil=0, mrt=False, nu=4e-3),
        # binary16 relative to the local velocity, an odd width
        dict(name="les2047x2048_fp16rel", kind="steps", nx=2047, ny=2048, steps=8, precision="fp16rel", delta=2.0,
             stencil=0, mrt=False, nu=4e-3),
        # the learned closure in the loop on the 256^2 LES grid
        dict(name="closure256_fp32", kind="closure", n=256, steps=64, precision="fp32", delta=2.0, nu=5e-3),
        # the parameter study: 48 runs of three sizes in one launch per step
        dict(name="ensemble48_fp32", kind="ensemble", sizes="128 512 1024", per_size=16, steps=32,
             precision="fp32", delta=2.0),
        # one whole short run as a batch job makes it, host fields in, host snapshot out
        dict(name="job2048_fp32", kind="job", nx=2048, ny=2048, steps=20, precision="fp32", delta=0.0, nu=2e-3),
        # one checkpoint of the LES-vs-DNS comparison: 2048^2 filtered to 1024^2
        dict(name="checkpoint2048_r2", kind="checkpoint", n=2048, r=2, precision="fp32"),
        # one snapshot of the closure's data set and its a-priori evaluation
        dict(name="apriori2048_r8", kind="apriori", n=2048, r=8, delta=2.0),
        # one training iteration's gradient: eight 256^2 snapshots
        dict(name="gradient8x256", kind="gradient", batch=8, h=256, w=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["steps", "steps", "steps", "closure", "ensemble", "job", "checkpoint", "apriori", "gradient"])
    if kind in ("steps", "job"):
        nx, ny = _log_int(rng, 48, 4096), _log_int(rng, 48, 4096)
        precision = rng.choice(["fp64", "fp32", "fp32", "fp16", "fp16rel"])
        most = 1.6e7 if precision == "fp64" else 1.2e8  # cell updates of a pass
        steps = max(1, min(_log_int(rng, 1, 64), int(most / (nx * ny))))
        c = dict(kind=kind, nx=nx, ny=ny, steps=steps, precision=precision, delta=rng.choice([0.0, 1.0, 2.0]),
                 nu=rng.uniform(4e-3, 2e-2))
        if kind == "steps":
            c.update(stencil=rng.randint(0, 1), mrt=rng.random() < 0.3)
        return c
    if kind == "closure":
        n = _log_int(rng, 48, 700)
        return dict(kind=kind, n=n, steps=max(1, min(_log_int(rng, 1, 64), int(8e6 / (n * n)))),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), delta=2.0, nu=rng.uniform(4e-3, 2e-2))
    if kind == "ensemble":
        sizes = [_log_int(rng, 40, 700) for _ in range(rng.randint(2, 4))]
        return dict(kind=kind, sizes=" ".join(str(s) for s in sizes), per_size=rng.randint(2, 6),
                    steps=_log_int(rng, 4, 40), precision=rng.choice(["fp32", "fp32", "fp16"]),
                    delta=rng.choice([1.0, 2.0]))
    if kind == "checkpoint":
        r = rng.choice([2, 4, 8])
        return dict(kind=kind, n=r * _log_int(rng, 48, min(1100, 4096 // r)), r=r,
                    precision=rng.choice(["fp32", "fp64"]))
    if kind == "apriori":
        r = rng.choice([2, 4, 8])
        return dict(kind=kind, n=r * _log_int(rng, 24, 2048 // r), r=r, delta=rng.choice([1.0, 2.0]))
    return dict(kind=kind, batch=rng.randint(1, 8), h=_log_int(rng, 16, 256), w=_log_int(rng, 16, 256))


# ------------------------------------------------------------------------------ inputs
def _modes(shape, h, w, kmax, gen, count=6):
    """Smooth random periodic fields [*shape, h, w] of unit variance: a few Fourier modes."""
    k = torch.randint(-kmax, kmax + 1, (2, *shape, count), generator=gen, device=DEVICE).double()
    ph = 2 * math.pi * torch.rand((*shape, count), generator=gen, device=DEVICE, dtype=torch.float64)
    a = torch.randn((*shape, count), generator=gen, device=DEVICE, dtype=torch.float64) * math.sqrt(2.0 / count)
    x = 2 * math.pi * torch.arange(w, device=DEVICE, dtype=torch.float64) / w
    y = 2 * math.pi * torch.arange(h, device=DEVICE, dtype=torch.float64) / h
    px, py = k[0][..., None] * x + ph[..., None], k[1][..., None] * y
    # sum_m a_m cos(px_m + py_m) as two products of [h, m] and [m, w]
    ca, sa = (a[..., None] * torch.cos(py)).transpose(-1, -2), (a[..., None] * torch.sin(py)).transpose(-1, -2)
    return ca @ torch.cos(px) - sa @ torch.sin(px)


def _fields(nx, ny, seed):
    """rho, ux, uy, bx, by [5, ny, nx]: a magnetized Kelvin-Helmholtz double shear layer with
    seeded amplitudes, perturbed by smooth modes and a little noise."""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    pick = random.Random(seed)
    u0, b0 = pick.uniform(0.03, 0.05), pick.uniform(0.01, 0.03)
    y = torch.arange(ny, device=DEVICE, dtype=torch.float64)[:, None]
    d = ny / 32.0
    f = _modes((5,), ny, nx, 4, gen)
    f *= torch.tensor([2e-3, 0.1 * u0, 0.1 * u0, 0.2 * b0, 0.2 * b0], device=DEVICE, dtype=torch.float64)[:, None, None]
    f[0] += 1.0
    f[1] += u0 * (torch.tanh((y - ny / 4.0) / d) - torch.tanh((y - 3.0 * ny / 4.0) / d) - 1.0)
    f[2] += 1e-5 * (2.0 * torch.rand((ny, nx), generator=gen, device=DEVICE, dtype=torch.float64) - 1.0)
    f[3] += b0
    return f


def _rates(case):
    """Nine fluid rates and the magnetic rate: the paper's single rate, or unequal ones."""
    s = 1.0 / (3.0 * case["nu"] + 0.5)
    rates = [s] * 9
    if case.get("mrt"):
        rates[5] = rates[6] = 1.5
        rates[7], rates[8] = 1.3, 1.4
    return rates, s


def _params(case, nx, ny):
    rates, s_m = _rates(case)
    return lbmhd.make_params(nx, ny, rates, s_m, case["delta"], PRECISION[case["precision"]],
                             case.get("stencil", 0))


def _network(seed):
    """Network parameters as training starts from (uniform +-1/sqrt(fan_in)), small biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for ci, co in ((12, 32), (32, 32), (32, 4)):
        parts += [rng.uniform(-1, 1, co * ci * 9) / math.sqrt(9 * ci), 0.02 * rng.uniform(-1, 1, co)]
    return np.concatenate(parts).astype(np.float32)


def _scales(n):
    """Channel scales of an n x n state: velocity, field and their differences across a shear
    layer n/32 wide; subgrid terms of the order of the squared differences."""
    g = 0.04 * 32.0 / n
    return (np.array([0.04, 0.02, 0.02, 0.01] + [0.2 * g, g, 0.2 * g, 0.2 * g] + [0.1 * g] * 4, np.float32),
            np.full(4, 0.1 * g * g, np.float32))


def _members(case, seed):
    """(parameters, size, seed) of the ensemble's members."""
    pick, out = random.Random(seed), []
    for n in (int(v) for v in case["sizes"].split()):
        for _ in range(case["per_size"]):
            out.append((dict(case, nu=pick.uniform(4e-3, 2e-2)), n, pick.randrange(1 << 30)))
    return out


def _batch(case, seed):
    """Scaled features [b, 12, h, w] and targets [b, 4, h, w] that depend on them."""
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    b, h, w = case["batch"], case["h"], case["w"]
    x = _modes((b, 12), h, w, 6, gen).float()
    t = (0.6 * torch.tanh(x[:, :4] + 0.5 * x[:, 4:8]) + 0.3 * x[:, 8:12] * x[:, :4]).contiguous()
    return x, t


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("steps", "closure"):
        nx, ny = (case["n"], case["n"]) if kind == "closure" else (case["nx"], case["ny"])
        f = _fields(nx, ny, seed)
        st = {"kind": kind, "steps": case["steps"], "dtype": SNAPSHOT[case["precision"]],
              "sim": lbmhd.Lbmhd(_params(case, nx, ny), *f, device=True), "out": torch.empty_like(f)}
        if kind == "closure":
            st["closure"] = lbmhd.Closure(_network(seed), *_scales(nx))
            st["closure"].attach(st["sim"].h)
        return st
    if kind == "ensemble":
        members, views, o = [], [], 0
        ms = _members(case, seed)
        out = torch.empty((5, sum(n * n for _, n, _ in ms)), dtype=torch.float64, device=DEVICE)
        for c, n, s in ms:
            members.append((_params(c, n, n), list(_fields(n, n, s).cpu().numpy())))
            views.append([out[k, o:o + n * n] for k in range(5)])
            o += n * n
        ens = lbmhd.Ensemble(members)
        return {"kind": kind, "steps": case["steps"], "dtype": SNAPSHOT[case["precision"]], "ens": ens,
                "views": views, "out": out, "stream": torch.cuda.ExternalStream(ens.stream)}
    if kind == "job":
        f = _fields(case["nx"], case["ny"], seed)
        host = torch.empty(f.shape, dtype=torch.float64, pin_memory=True)
        host.copy_(f)
        snap = torch.empty(f.shape, dtype=SNAPSHOT[case["precision"]], pin_memory=True)
        return {"kind": kind, "steps": case["steps"], "dtype": snap.dtype, "params": _params(case, case["nx"], case["ny"]),
                "fields": list(host.numpy()), "host": host, "snap": snap, "out": torch.empty_like(f)}
    if kind == "checkpoint":
        n, r = case["n"], case["r"]
        m = n // r
        f = _fields(n, n, seed)
        p = lbmhd.lbmhd_params_srt(n, n, 2e-3, 2e-3, 0.0, PRECISION[case["precision"]])
        nb = m // 2 + 1
        new = lambda *s: torch.empty(s, dtype=torch.float64, device=DEVICE)  # noqa: E731
        return {"kind": kind, "r": r, "nb": nb, "sim": lbmhd.Lbmhd(p, *f, device=True), "fine": list(f.clone()),
                "coarse": [new(m, m) for _ in range(5)], "ek": new(nb), "em": new(nb),
                "work": torch.empty(lbmhd.lbmhd_energy_spectrum_work_bytes(m), dtype=torch.uint8, device=DEVICE)}
    if kind == "apriori":
        n, r = case["n"], case["r"]
        m = n // r
        f32 = lambda c: torch.empty((1, c, m, m), dtype=torch.float32, device=DEVICE)  # noqa: E731
        return {"kind": kind, "r": r, "delta": case["delta"], "fine": _fields(n, n, seed),
                "closure": lbmhd.Closure(_network(seed), *_scales(m)), "x": f32(12), "t": f32(4), "y": f32(4),
                "work": torch.empty(9 * m * m, dtype=torch.float64, device=DEVICE)}
    x, t = _batch(case, seed)
    return {"kind": kind, "x": x, "t": t,
            "closure": lbmhd.Closure(_network(seed), np.ones(12, np.float32), np.ones(4, np.float32))}


# ------------------------------------------------------------------------------ one pass
def run(state):
    kind = state["kind"]
    if kind in ("steps", "closure"):
        state["sim"].step(state["steps"])
        state["sim"].moments_device(list(state["out"]))
        return list(state["out"].to(state["dtype"]))
    if kind == "ensemble":
        ens, here = state["ens"], torch.cuda.current_stream()
        ens.step(state["steps"])
        state["stream"].wait_stream(here)  # the snapshot buffer is read on this stream
        for i, views in enumerate(state["views"]):
            lbmhd.lbmhd_moments_device(ens.member(i), views)
        here.wait_stream(state["stream"])
        return list(state["out"].to(state["dtype"]))
    if kind == "job":
        with lbmhd.Lbmhd(state["params"], *state["fields"]) as sim:
            sim.step(state["steps"])
            sim.moments_device(list(state["out"]))
            state["snap"].copy_(state["out"].to(state["dtype"]), non_blocking=True)
            torch.cuda.current_stream().synchronize()  # the host reads the snapshot
        return list(state["snap"])
    if kind == "checkpoint":
        state["sim"].moments_device(state["fine"])
        for a, b in zip(state["fine"], state["coarse"]):
            lbmhd.lbmhd_block_mean_device(a, state["r"], b)
        lbmhd.lbmhd_energy_spectrum_device(*state["coarse"][1:], state["nb"], state["ek"], state["em"], state["work"])
        return {"coarse": state["coarse"], "e_kin": state["ek"], "e_mag": state["em"],
                "diagnostics": state["sim"].diagnostics()}
    if kind == "apriori":
        c = state["closure"]
        c.training_pair(state["fine"], state["r"], state["delta"], state["x"][0], state["t"][0], state["work"])
        c.forward(state["x"], state["y"], tensor_cores=True)
        return [state["x"], state["t"], state["y"]]
    loss, grad = state["closure"].gradient(state["x"], state["t"])
    return {"loss": loss, "grad": grad}


def work(case):
    """What one pass cannot do without.  A time step reads the stored state and writes the next;
    a snapshot reads the state and writes five binary64 fields."""
    kind = case["kind"]
    if kind in ("steps", "closure", "ensemble", "job"):
        if kind == "ensemble":
            cells = case["per_size"] * sum(int(v) ** 2 for v in case["sizes"].split())
        else:
            cells = case["n"] ** 2 if kind == "closure" else case["nx"] * case["ny"]
        state = cells * PLANES[case["precision"]] * ELEM[case["precision"]]
        k = case["steps"]
        flops = cells * k * (FLOPS_STEP + (FLOPS_NET if kind == "closure" else 0))
        return {"bytes": 2 * k * state + state + 40 * cells + (40 * cells if kind == "job" else 0), "flops": flops}
    if kind == "checkpoint":
        n2, m2 = case["n"] ** 2, (case["n"] // case["r"]) ** 2
        state = n2 * 27 * ELEM[case["precision"]]
        return {"bytes": state + 40 * n2 + 40 * m2, "flops": 100 * n2 + 10 * m2 * math.log2(m2)}
    if kind == "apriori":
        n2, m2 = case["n"] ** 2, (case["n"] // case["r"]) ** 2
        return {"bytes": 40 * n2 + 80 * m2, "flops": 40 * n2 + FLOPS_NET * m2}
    cells = case["batch"] * case["h"] * case["w"]
    # forward, weight gradients, and data gradients of all layers but the first
    return {"bytes": 64 * cells, "flops": cells * (3 * FLOPS_NET - 2 * 9 * 12 * 32)}


# ------------------------------------------------------------------------------ plain binary64
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _shift(a, dx, dy):
    """a(x + dx, y + dy), periodic."""
    return torch.roll(a, (-dy, -dx), (-2, -1))


def _diff(a, axis, stencil):
    """d_x (axis 0) or d_y (axis 1): central two-point, or isotropic over the nine neighbours."""
    if not stencil:
        e = (1, 0) if axis == 0 else (0, 1)
        return 0.5 * (_shift(a, *e) - _shift(a, -e[0], -e[1]))
    out = torch.zeros_like(a)
    for i in range(1, 9):
        c = (CX, CY)[axis][i]
        if c:
            out += 3.0 * WT[i] * c * _shift(a, CX[i], CY[i])
    return out


def _equilibrium(f):
    """Populations (f_i - w_i, g_x, g_y; each [9, ny, nx]) of the fields without subgrid terms."""
    rho, u, v, b, d = f
    pf, px, py = [], [], []
    for i in range(9):
        cu, cb, cc = CX[i] * u + CY[i] * v, CX[i] * b + CY[i] * d, CX[i] ** 2 + CY[i] ** 2
        pf.append(WT[i] * ((rho - 1) + rho * (3 * cu + 4.5 * cu * cu - 1.5 * (u * u + v * v))
                           + 4.5 * (0.5 * (b * b + d * d) * cc - cb * cb)))
        px.append(WT[i] * (b + 3 * (cu * b - cb * u)))
        py.append(WT[i] * (d + 3 * (cu * d - cb * v)))
    return pf, px, py


def _macro(pf, px, py):
    j = [sum(c[i] * pf[i] for i in range(9) if c[i]) for c in (CX, CY)]
    return 1 + sum(pf), j[0], j[1], sum(px), sum(py)


def _moment_rows():
    """Rows 3..8 of the fluid transform as polynomials of the lattice velocities."""
    x, y = np.array(CX, float), np.array(CY, float)
    r2 = x * x + y * y
    return {3: x * y, 4: x * x - y * y, 5: (3 * r2 - 5) * x, 6: (3 * r2 - 5) * y,
            7: np.where(r2 == 0, 4.0, np.where(r2 == 1, -5.0, 4.0)), 8: np.where(r2 == 0, 4.0, np.where(r2 == 1, 0.0, -1.0))}


def _advance(pop, case, corr=None):
    """One step: collide toward the filtered equilibria, then stream."""
    pf, px, py = pop
    rates, s_m = _rates(case)
    st, k = case.get("stencil", 0), case["delta"] ** 2 / 12.0
    rho, jx, jy, bx, by = _macro(pf, px, py)
    gj = [[_diff(a, ax, st) for ax in (0, 1)] for a in (jx, jy)]
    gb = [[_diff(a, ax, st) for ax in (0, 1)] for a in (bx, by)]
    dot = lambda p, q: p[0] * q[0] + p[1] * q[1]  # noqa: E731
    sxx, syy = (jx * jx + k * dot(gj[0], gj[0])) / rho, (jy * jy + k * dot(gj[1], gj[1])) / rho
    sxy = (jx * jy + k * dot(gj[0], gj[1])) / rho - (bx * by + k * dot(gb[0], gb[1]))
    mxx, myy = bx * bx + k * dot(gb[0], gb[0]), by * by + k * dot(gb[1], gb[1])
    e = (jx * by - jy * bx + k * (dot(gj[0], gb[1]) - dot(gj[1], gb[0]))) / rho
    nrm, trc = (sxx - syy) - (mxx - myy), sxx + syy
    if corr is not None:
        sxy, nrm, trc, e = sxy + corr[0], nrm + corr[1], trc + corr[2], e + corr[3]
    eq = {3: sxy, 4: nrm, 5: -jx, 6: -jy, 7: -3 * trc, 8: 5 / 3 * (rho - 1) - 3 * trc}
    new = [p.clone() for p in pf]
    for m, row in _moment_rows().items():
        n = sum(float(row[i]) * pf[i] for i in range(9) if row[i]) - eq[m]
        n *= rates[m] / float((row * row).sum())
        for i in range(9):
            if row[i]:
                new[i] -= float(row[i]) * n
    nxp = [px[i] + s_m * (WT[i] * (bx - 3 * CY[i] * e) - px[i]) for i in range(9)]
    nyp = [py[i] + s_m * (WT[i] * (by + 3 * CX[i] * e) - py[i]) for i in range(9)]
    return tuple([_shift(p[i], -CX[i], -CY[i]) for i in range(9)] for p in (new, nxp, nyp))


def _read(pop):
    rho, jx, jy, bx, by = _macro(*pop)
    return [rho, jx / rho, jy / rho, bx, by]


def _layers(theta):
    out, o = [], 0
    for ci, co in ((12, 32), (32, 32), (32, 4)):
        out.append((theta[o:o + co * ci * 9].reshape(co, ci, 3, 3), theta[o + co * ci * 9:o + co * ci * 9 + co]))
        o += co * ci * 9 + co
    return out


def _net(theta, x):
    for n, (w, b) in enumerate(_layers(theta)):
        y = b[None, :, None, None]
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                y = y + torch.einsum("oc,bchw->bohw", w[:, :, dy + 1, dx + 1], _shift(x, dx, dy))
        x = torch.tanh(y) if n < 2 else y
    return x


def _features(u, v, b, d, in_scale):
    ch = [u, v, b, d] + [_diff(a, ax, 0) for a in (u, v, b, d) for ax in (0, 1)]
    return torch.stack(ch) / torch.tensor(in_scale, dtype=torch.float64, device=DEVICE)[:, None, None]


def _box(a, r):
    return a.reshape(a.shape[-2] // r, r, a.shape[-1] // r, r).mean((1, 3))


def _spectra(u, v, b, d, nb):
    n = u.shape[0]
    k = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=DEVICE)
    shell = torch.floor(torch.sqrt(k[:, None] ** 2 + k[None, :] ** 2) + 0.5).long().flatten()
    power = [(torch.fft.fft2(a).abs() / n ** 2) ** 2 for a in (u, v, b, d)]
    return [torch.bincount(shell, 0.5 * (p + q).flatten(), minlength=n)[:nb] for p, q in (power[:2], power[2:])]


def _diagnostics(rho, u, v, b, d):
    dx = [_diff(a, 0, 1) for a in (b, d)]
    dy = [_diff(a, 1, 1) for a in (b, d)]
    vals = [rho.sum(), (rho * u).sum(), (rho * v).sum(), b.sum(), d.sum(), (0.5 * rho * (u * u + v * v)).sum(),
            (0.5 * (b * b + d * d)).sum(), (dx[0] + dy[1]).abs().max(), (_diff(b, 0, 0) + _diff(d, 1, 0)).abs().max(),
            torch.stack(dx + dy).abs().max()]
    return torch.stack(vals)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("steps", "closure", "job"):
        nx, ny = (case["n"], case["n"]) if kind == "closure" else (case["nx"], case["ny"])
        pop = _equilibrium(_fields(nx, ny, seed))
        if kind == "closure":
            theta = torch.tensor(_network(seed), dtype=torch.float64, device=DEVICE)
            in_s, out_s = _scales(nx)
        for _ in range(case["steps"]):
            corr = None
            if kind == "closure":
                _, u, v, b, d = _read(pop)
                corr = _net(theta, _features(u, v, b, d, in_s)[None])[0]
                corr = corr * torch.tensor(out_s, dtype=torch.float64, device=DEVICE)[:, None, None]
            pop = _advance(pop, case, corr)
        return _read(pop)
    if kind == "ensemble":
        out = []
        for c, n, s in _members(case, seed):
            pop = _equilibrium(_fields(n, n, s))
            for _ in range(case["steps"]):
                pop = _advance(pop, c)
            out.append(torch.stack([a.flatten() for a in _read(pop)]))
        return list(torch.cat(out, 1))
    if kind == "checkpoint":
        f = _fields(case["n"], case["n"], seed)
        coarse = [_box(a, case["r"]) for a in f]
        ek, em = _spectra(*coarse[1:], coarse[0].shape[0] // 2 + 1)
        return {"coarse": coarse, "e_kin": ek, "e_mag": em, "diagnostics": _diagnostics(*f)}
    if kind == "apriori":
        rho, u, v, b, d = _fields(case["n"], case["n"], seed)
        r, k = case["r"], case["delta"] ** 2 / 12.0
        in_s, out_s = _scales(case["n"] // r)
        R, X, Y, B, D = (_box(a, r) for a in (rho, rho * u, rho * v, b, d))
        true = [_box(rho * u * v - b * d, r) - (X * Y / R - B * D),
                _box(rho * (u * u - v * v) - (b * b - d * d), r) - ((X * X - Y * Y) / R - (B * B - D * D)),
                _box(rho * (u * u + v * v), r) - (X * X + Y * Y) / R, _box(u * d - v * b, r) - (X * D - Y * B) / R]
        gx, gy, gb, gd = ([_diff(a, ax, 0) for ax in (0, 1)] for a in (X, Y, B, D))
        dot = lambda p, q: p[0] * q[0] + p[1] * q[1]  # noqa: E731
        model = [k * (dot(gx, gy) / R - dot(gb, gd)), k * ((dot(gx, gx) - dot(gy, gy)) / R - dot(gb, gb) + dot(gd, gd)),
                 k * (dot(gx, gx) + dot(gy, gy)) / R, k * (dot(gx, gd) - dot(gy, gb)) / R]
        x = _features(X / R, Y / R, B, D, in_s)[None]
        t = torch.stack([(p - q) / float(s) for p, q, s in zip(true, model, out_s)])[None]
        return [x, t, _net(torch.tensor(_network(seed), dtype=torch.float64, device=DEVICE), x)]
    x, t = _batch(case, seed)
    theta = torch.tensor(_network(seed), dtype=torch.float64, device=DEVICE, requires_grad=True)
    loss = 0.5 * ((_net(theta, x.double()) - t.double()) ** 2).mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": theta.grad}
