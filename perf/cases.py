"""Performance cases of the SPFM library: the calls a study makes, over the range of its grids.

A case is one call of the public binding (``paper_1910_05180_gb300.spfm``) on fields that sit on
the device:

- ``step``: ``Grid.step``, n explicit steps of one grid (TI_<hkl>, TI_n or CF; FP64, FP32 or BF16
  storage; periodic, contact-angle or no-flux faces; round to nearest or stochastic);
- ``batch``: ``Batch.step``, n steps of many grids together (orientation sweeps, served jobs);
- ``relax``: ``Grid.step_conserving``, n steps at constant particle volume;
- ``stats``: ``Grid.stats``, the FP64 interface diagnostics.

The fields are the ideal profiles the studies start from (planes, grains, cubes), placed at a
seeded sub-cell offset; driving forces are of the studies' size, small enough that the interface
stays inside its grid over many calls.  ``exact`` restates the discrete equations in plain FP64
torch.
"""
import math

import numpy as np
import torch

from paper_1910_05180_gb300 import spfm as S

DTYPE = {"f64": S.SPFM_F64, "f32": S.SPFM_F32, "bf16": S.SPFM_BF16}
SCHEME = {"ti": S.SPFM_TI_GLOBAL, "tin": S.SPFM_TI_LOCAL, "cf": S.SPFM_FD}
BYTES = {"f64": 8, "f32": 4, "bf16": 2}
P, N, C = S.SPFM_PERIODIC, S.SPFM_NOFLUX, S.SPFM_CONTACT
FACES = {"periodic": (P,) * 6, "contact": (C,) * 6, "channel": (N, N, P, P, P, P)}
AXES = {"100": (1.0, 0.0, 0.0), "111": (1.0, 1.0, 1.0), "120": (1.0, 2.0, 0.0)}
MAX_CELL_STEPS = 512 ** 3 * 8   # cell updates of the largest listed step case


def listed():
    return [
        # a small velocity-measurement job, stepped and looked at every few steps: launch latency
        dict(name="job_32_f32", op="step", nx=32, ny=32, nz=32, dtype="f32", scheme="ti", stencil=26, lam=4.0,
             faces="contact", shape="plane", n="random", rounding="stochastic", dt=0.05, steps=10),
        # planar interface in a channel (no-flux along x, periodic across), FP64, 7-point
        dict(name="plane_128x32x32_f64", op="step", nx=128, ny=32, nz=32, dtype="f64", scheme="ti", stencil=6,
             lam=4.0, faces="channel", shape="plane", n="100", rounding="nearest", dt=0.1, steps=20),
        # a ragged single job of the serving range with a random normal
        dict(name="job_ragged_f32", op="step", nx=150, ny=133, nz=117, dtype="f32", scheme="ti", stencil=26, lam=5.0,
             faces="contact", shape="plane", n="random", rounding="nearest", dt=0.05, steps=20),
        # tilted plane through a box, contact-angle faces, FP32 and FP64 storage
        dict(name="tilted_256_f32", op="step", nx=256, ny=256, nz=256, dtype="f32", scheme="ti", stencil=26, lam=3.0,
             faces="contact", shape="plane", n="111", rounding="nearest", dt=0.05, steps=10),
        dict(name="tilted_256_f64", op="step", nx=256, ny=256, nz=256, dtype="f64", scheme="ti", stencil=26, lam=3.0,
             faces="contact", shape="plane", n="111", rounding="nearest", dt=0.05, steps=3),
        # the large curved grain, FP32 and BF16 storage
        dict(name="grain_512_f32", op="step", nx=512, ny=512, nz=512, dtype="f32", scheme="ti", stencil=26, lam=3.0,
             faces="periodic", shape="sphere", n="120", rounding="nearest", dt=0.05, steps=8),
        dict(name="grain_384_bf16", op="step", nx=384, ny=384, nz=384, dtype="bf16", scheme="ti", stencil=26, lam=3.0,
             faces="periodic", shape="sphere", n="120", rounding="stochastic", dt=0.05, steps=8),
        # the grain under the local-normal model
        dict(name="grain_320_tin", op="step", nx=320, ny=320, nz=320, dtype="f32", scheme="tin", stencil=26, lam=3.0,
             faces="periodic", shape="sphere", n="120", rounding="nearest", dt=0.05, steps=4),
        # an orientation sweep: grids of 32 to 96 cells a side, random normals
        dict(name="sweep_64_f32", op="batch", grids=64, edge_lo=32, edge_hi=96, dtype="f32", scheme="ti", stencil=26,
             faces="contact", rounding="nearest", dt=0.05, steps=16),
        # a window of served jobs: 32 to 192 cells a side, stochastic rounding
        dict(name="served_32_f32", op="batch", grids=32, edge_lo=32, edge_hi=192, dtype="f32", scheme="ti",
             stencil=26, faces="contact", rounding="stochastic", dt=0.05, steps=16),
        # cube relaxing to a sphere at constant volume
        dict(name="relax_60_tin", op="relax", nx=60, ny=60, nz=60, dtype="f32", scheme="tin", stencil=26, lam=4.0,
             faces="periodic", shape="cube", n="120", rounding="nearest", dt=0.05, steps=10),
        # the diagnostics of the large grain
        dict(name="stats_512_f32", op="stats", nx=512, ny=512, nz=512, dtype="f32", lam=3.0, faces="periodic",
             shape="sphere", n="120"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step"] * 5 + ["batch"] * 2 + ["relax", "stats"])
    rounding = rng.choice(["nearest", "stochastic"])
    if op == "batch":
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        lo = _log_int(rng, 24, 64)
        hi = max(lo + 8, _log_int(rng, 48, 192 if dtype == "f32" else 64))
        most = 8 if dtype == "f64" else (64 if hi <= 100 else 24)
        return dict(op="batch", grids=rng.randint(2, most), edge_lo=lo, edge_hi=hi, dtype=dtype,
                    scheme=rng.choice(["ti", "ti", "cf"]), stencil=26,
                    faces=rng.choice(["contact", "contact", "channel"]),
                    rounding=rounding if dtype == "f32" else "nearest", dt=0.05, steps=rng.choice([5, 16, 20]))
    if op == "relax":
        edge = rng.randint(40, 97)
        dtype = rng.choice(["f32", "f32", "f64"])
        return dict(op="relax", nx=edge, ny=edge + rng.randint(0, 5), nz=edge, dtype=dtype,
                    scheme=rng.choice(["ti", "cf"] + (["tin"] if dtype == "f32" else [])), stencil=26,
                    lam=rng.choice([3.0, 4.0]), faces="periodic", shape="cube", n="120", rounding="nearest",
                    dt=0.05, steps=rng.randint(5, 12))
    if op == "stats":
        edge = _log_int(rng, 32, 448)
        return dict(op="stats", nx=edge, ny=max(24, edge + rng.randint(-9, 9)), nz=max(24, edge + rng.randint(-9, 9)),
                    dtype=rng.choice(["f32", "f32", "f64", "bf16"]), lam=rng.choice([2.0, 3.0, 4.0, 6.0]),
                    faces="periodic", shape=rng.choice(["sphere", "plane"]), n="random")
    dtype = rng.choice(["f32", "f32", "f32", "f64", "bf16"])
    scheme = rng.choice(["ti", "ti", "ti", "tin", "cf"])
    faces = rng.choice(["contact", "periodic", "channel"])
    top = 96 if dtype == "f64" and scheme == "tin" else (224 if dtype == "f64" else 448)
    shape = [max(24, int(_log_int(rng, 32, top) * rng.uniform(0.8, 1.0))) for _ in range(3)]
    # a cell update of TI_n or in FP64 takes many times that of the listed grain
    weight = (8 if scheme == "tin" else 1) * (20 if dtype == "f64" else 1)
    steps = min(rng.randint(4, 20), max(1, MAX_CELL_STEPS // (shape[0] * shape[1] * shape[2] * weight)))
    if faces == "periodic" and rng.random() < 0.6:
        shape[0] = max(32, shape[0] // 32 * 32)
    return dict(op="step", nx=shape[0], ny=shape[1], nz=shape[2], dtype=dtype, scheme=scheme,
                stencil=rng.choice([26, 26, 26, 18, 6]), lam=rng.choice([3.0, 4.0, 5.0, 6.0]), faces=faces,
                shape="sphere" if faces == "periodic" else "plane",
                n=rng.choice(["random", "random", "111", "120"]) if faces != "channel" else "100",
                rounding="stochastic" if dtype == "bf16" else (rounding if dtype == "f32" else "nearest"), dt=0.05,
                steps=steps)


# ---------------------------------------------------------------- inputs


def _unit(v):
    v = np.asarray(v, dtype=np.float64)
    return v / np.linalg.norm(v)


def _normal(case, rng):
    return tuple(float(x) for x in (_unit(rng.normal(size=3)) if case["n"] == "random" else _unit(AXES[case["n"]])))


def _spec(case, rng):
    """One grid's seeded parameters: normal, profile offset, driving force."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    mid = [(d - 1) / 2.0 + float(rng.uniform(-0.5, 0.5)) for d in (nx, ny, nz)]
    n = _normal(case, rng)
    R = 0.293 * min(nx, ny, nz)
    if case["shape"] == "sphere":
        dF = 2.0 / R   # balances the grain's curvature
    else:
        dF = float(np.exp(rng.uniform(np.log(1e-4), np.log(2e-3)))) * float(rng.choice([-1.0, 1.0]))
    return dict(nx=nx, ny=ny, nz=nz, n=n, mid=mid, c=float(np.dot(n, mid)), R=R, half=0.2 * nx,
                dF=0.0 if case["op"] == "relax" else dF, lam=case["lam"], faces=FACES[case["faces"]],
                shape=case["shape"], seed=int(rng.integers(1 << 31)))


def _specs(case, seed):
    rng = np.random.default_rng(seed)
    if case["op"] != "batch":
        return [_spec(case, rng)]
    out = []
    sizes = np.random.default_rng(case["grids"])   # a batch's sizes are the case's, not the seed's
    for _ in range(case["grids"]):
        edge = case["edge_lo"] + int(sizes.integers((case["edge_hi"] - case["edge_lo"]) // 16 + 1)) * 16
        one = dict(case, nx=edge, ny=edge, nz=edge, lam=float(rng.choice([2.0, 3.0, 4.0, 6.0])), shape="plane",
                   n="100" if case["faces"] == "channel" else "random")
        out.append(_spec(one, rng))
    return out


def _profile(sp, dtype, device):
    """The ideal profile (FP64, rounded once to the storage type), dense (nz, ny, nx)."""
    x, y, z = (torch.arange(d, dtype=torch.float64, device=device) for d in (sp["nx"], sp["ny"], sp["nz"]))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    lam, mid = sp["lam"], sp["mid"]
    if sp["shape"] == "plane":
        d = x * sp["n"][0] + y * sp["n"][1] + z * sp["n"][2] - sp["c"]
        phi = 0.5 * (1.0 - torch.tanh(2.0 * d / lam))
    elif sp["shape"] == "sphere":
        r = ((x - mid[0]) ** 2 + (y - mid[1]) ** 2 + (z - mid[2]) ** 2).sqrt()
        phi = 0.5 * (1.0 - torch.tanh(2.0 * (sp["R"] - r) / lam))
    else:
        phi = 1.0
        for p, m in ((x, mid[0]), (y, mid[1]), (z, mid[2])):
            phi = phi * (0.5 * (1.0 - torch.tanh(2.0 * ((p - m).abs() - sp["half"]) / lam)))
        phi = 1.0 - phi
    return phi.to(S.TORCH_DTYPE[DTYPE[dtype]])


def _grid(sp, case, stream):
    g = S.Grid(sp["nx"], sp["ny"], sp["nz"], dtype=DTYPE[case["dtype"]], bc=sp["faces"], n=sp["n"],
               center=tuple(sp["mid"]), stream=stream)
    if case.get("rounding") == "stochastic":
        g.set_rounding(S.SPFM_ROUND_STOCHASTIC, seed=sp["seed"])
    if case["op"] == "stats":
        g.init_planar(sp["c"], sp["lam"])   # the diagnostics use the model of the last init or step
    g.set_field(_profile(sp, case["dtype"], "cuda"))
    return g


def _kw(sp, case):
    return dict(lam=sp["lam"], dt=case["dt"], stencil=case["stencil"], scheme=SCHEME[case["scheme"]])


def prepare(case, seed):
    specs = _specs(case, seed)
    stream = torch.cuda.Stream() if case["op"] == "batch" else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        grids = [_grid(sp, case, stream) for sp in specs]
        state = dict(case=case, grids=grids)
        if case["op"] == "batch":
            state["batch"] = S.Batch(grids, stream=stream)
            state["args"] = [S.step_args(dF=sp["dF"], **_kw(sp, case)) for sp in specs]
        elif case["op"] != "stats":
            state["kw"] = _kw(specs[0], case)
            if case["op"] == "step":
                state["kw"]["dF"] = specs[0]["dF"]
    torch.cuda.synchronize()
    return state


def run(state):
    case, grids = state["case"], state["grids"]
    if case["op"] == "step":
        grids[0].step(case["steps"], **state["kw"])
    elif case["op"] == "batch":
        state["batch"].step(case["steps"], state["args"])
    elif case["op"] == "relax":
        grids[0].step_conserving(case["steps"], **state["kw"])
    else:
        return grids[0].stats()
    return [g.current() for g in grids]


def work(case):
    """One read and one write of every cell per step (stats: one read); arithmetic of one cell update."""
    if case["op"] == "batch":
        cells = sum(sp["nx"] ** 3 for sp in _specs(case, 0))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    size = BYTES[case["dtype"]]
    if case["op"] == "stats":
        return {"bytes": cells * size, "flops": cells * 4}
    steps = case["steps"]
    per = {6: 12, 18: 28, 26: 36}[case["stencil"]] + {"cf": 8, "ti": 16, "tin": 120}[case["scheme"]]
    return {"bytes": cells * steps * 2 * size, "flops": cells * steps * per}


# ---------------------------------------------------------------- FP64 restatement


DIRS = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, -1, 0), (0, 1, -1), (1, 0, -1),
        (1, 1, 1), (-1, 1, 1), (1, -1, 1), (1, 1, -1)]
GAMMA = {6: (1.0, 0.0, 0.0), 18: (1 / 3, 2 / 3, 0.0), 26: (1 / 2, 1 / 3, 1 / 6)}
NDIRS = {6: 3, 18: 9, 26: 13}


def _padded(phi, sp):
    """The field with its ghost layer: x faces, then y, then z (periodic, copied, or shifted by Eq. 7)."""
    for ax, dim in ((0, 2), (1, 1), (2, 0)):
        m = phi.shape[dim]
        lo, hi = phi.narrow(dim, 0, 1), phi.narrow(dim, m - 1, 1)
        bc = sp["faces"][2 * ax]
        if bc == P:
            lo, hi = hi, lo
        elif bc == C:
            a = math.tanh(2.0 * sp["n"][ax] / sp["lam"])
            lo = (1 + a) * lo / (1 + a * (2 * lo - 1))
            hi = (1 - a) * hi / (1 - a * (2 * hi - 1))
        phi = torch.cat((lo, phi, hi), dim)
    return phi


def _shifted(p, d):
    z, y, x = (n - 2 for n in p.shape)
    return p[1 + d[2]:1 + d[2] + z, 1 + d[1]:1 + d[1] + y, 1 + d[0]:1 + d[0] + x]


def _rate(phi, sp, stencil, scheme, dF):
    """R_p of Eq. 2 in FP64 (M = Gamma = dx = 1, C_Gamma = 2/3)."""
    lam, nd = sp["lam"], NDIRS[stencil]
    shell = [sum(abs(x) for x in d) for d in DIRS]
    w = [GAMMA[stencil][s - 1] * (1.0, 0.5, 0.75)[s - 1] for s in shell]
    p = _padded(phi, sp)
    q, s = phi * (1 - phi), 1 - 2 * phi
    out = q * (-4.0 * dF / lam)
    for k in range(nd):
        out += (w[k] / shell[k]) * (_shifted(p, DIRS[k]) + _shifted(p, [-x for x in DIRS[k]]) - 2 * phi)
    cf = -(16.0 / 3.0) / lam ** 2 * sum(w[:nd])
    if scheme == "cf":
        return out.add_(q * s, alpha=cf)
    if scheme == "ti":
        pot, u = torch.zeros_like(phi), s * s
        for k in range(nd):
            A = math.tanh(2.0 * sum(a * b for a, b in zip(DIRS[k], sp["n"])) / lam) ** 2
            pot += (4.0 * w[k] / shell[k] * A) / (1 - A * u)
        return out.sub_(q * s * pot)
    psi = p.clamp(1e-6, 1 - 1e-6)
    psi = (0.25 * lam) * torch.log((1 - psi) / psi)
    g = [0.5 * (_shifted(psi, d) - _shifted(psi, [-x for x in d])) for d in DIRS[:3]]
    del psi, p
    norm = (g[0] ** 2 + g[1] ** 2 + g[2] ** 2).sqrt()
    flat = norm < 1e-8
    g = [x / torch.where(flat, 1.0, norm) for x in g]
    pot = torch.zeros_like(phi)
    for k in range(nd):
        A = torch.tanh((2.0 / lam) * sum(x * c for x, c in zip(g, DIRS[k]) if c)) ** 2
        pot += (4.0 * w[k] / shell[k]) * A / (1 - A * s * s)
    return out.sub_(q * s * torch.where(flat, -cf, pot))


def _sums(phi, sp):
    """The diagnostics of Sec. 2.3 over the band 1e-6 < phi < 1 - 1e-6."""
    x, y, z = (torch.arange(d, dtype=torch.float64, device=phi.device) for d in (sp["nx"], sp["ny"], sp["nz"]))
    band = ((phi > 1e-6) & (phi < 1 - 1e-6)).nonzero(as_tuple=True)
    v = phi[band]
    at = [x[band[2]], y[band[1]], z[band[0]]]
    q, psi = v * (1 - v), 0.25 * sp["lam"] * (torch.log1p(-v) - torch.log(v))
    pn = sum(a * b for a, b in zip(at, sp["n"]))
    r = sum((a - b) ** 2 for a, b in zip(at, sp["mid"])).sqrt()
    S_w, S_c, S_r = float(q.sum()), float((q * (pn - psi)).sum()), float((q * (r + psi)).sum())
    return dict(volume=float(phi.sum()), S_w=S_w, S_c=S_c, S_r=S_r, phi_min=float(phi.min()),
                phi_max=float(phi.max()), nonfinite=0.0, position=S_c / S_w, radius=S_r / S_w, energy=float("nan"),
                steps=0.0, time=0.0)


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    out = []
    for sp in _specs(case, seed):
        phi = _profile(sp, case["dtype"], device).double()
        if case["op"] == "stats":
            return _sums(phi, sp)
        for _ in range(case["steps"]):
            if case["op"] == "relax":
                rate = _rate(phi, sp, case["stencil"], case["scheme"], 0.0)
                q = phi * (1 - phi)
                phi = phi + case["dt"] * rate - (case["dt"] * rate.sum() / q.sum()) * q
            else:
                phi = phi + case["dt"] * _rate(phi, sp, case["stencil"], case["scheme"], sp["dF"])
        out.append(phi)
    return out
