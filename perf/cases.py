"""Performance cases of the dose library: what a treatment-planning program has it do.

Every case is one pass through the public entry points on seeded pencil-beam
matrices (proton spots on a lateral lattice, a Gaussian across the beam, a Bragg
curve along it; most voxels see no spot, the others see tens to thousands).  The
lattices, grids, spacings and truncation thresholds are those of this
repository's configurations (the 32x32x20 tiny beam, the 256x256x160 clinical
beam, the scenario matrices, the three-beam plan, the beam shaped like the
paper's liver beam 1) or lie between them, odd sizes among them.  The matrices
are made on the GPU from the seed, so that preparing a case is mostly the
library's own create call.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2103_09683_gb300 as dose

# The spot spacing, Gaussian width and truncation threshold of the clinical beam.
CLINICAL = dict(dx=1.25, dy=1.25, sigma=4.0, tau=0.009134)
# ... of the tiny beam (32 voxels across, 25 x 20 spots).
TINY = dict(dx=1.28, dy=1.6, sigma=3.0, tau=0.2423)
# ... of the beam shaped like the paper's liver beam 1: spots a quarter voxel apart.
LIVER = dict(dx=0.25, dy=0.25, sigma=4.0, tau=0.028798)

VALUE_BYTES = {"u16": 2, "bf16": 2, "f16": 2, "fp8": 1, "f32": 4}
VALUE_DTYPE = {"u16": torch.int16, "bf16": torch.int16, "f16": torch.int16, "fp8": torch.uint8, "f32": torch.int32}


def _case(name, op, fmt, grid, lattice, model, **more):
    c = dict(name=name, op=op, fmt=fmt, nx=grid[0], ny=grid[1], nz=grid[2], sx=lattice[0], sy=lattice[1], **model)
    c.update(more)
    return c


def listed():
    return [
        # The smallest call: one dose of the tiny beam (a planning program's
        # interactive re-evaluation of a few spots); launches and latency count.
        _case("dose_tiny", "dose", "bf16", (32, 32, 20), (25, 20), TINY),
        # A whole small optimisation: 100 projected-gradient steps captured in one
        # CUDA graph, the loop that the tiny configuration stands for.
        _case("pg100_tiny", "pg", "u16", (32, 32, 20), (25, 20), TINY, iters=100),
        # One dose evaluation of the clinical beam: the headline call.
        _case("dose_clinical", "dose", "u16", (256, 256, 160), (80, 50), CLINICAL),
        # Dose, objective and gradient in one pass: what an optimiser calls every
        # iteration, on the middle scenario beam.
        _case("objective_mid", "objective", "u16", (200, 200, 120), (50, 50), CLINICAL),
        # The same with FP8 values and row scales on an odd grid whose row count is
        # no multiple of 4.
        _case("objective_odd_fp8", "objective", "fp8", (161, 147, 83), (37, 29), CLINICAL),
        # A caller's own objective through autograd: forward dose, then the adjoint
        # of the caller's residual.
        _case("autograd_odd_bf16", "autograd", "bf16", (171, 155, 91), (41, 31), CLINICAL),
        # Three setup-shift scenarios of a beam times 16 spot-weight vectors in one
        # launch: uncertainty evaluation of a set of candidate plans.
        _case("batched_3x16", "batched", "u16", (160, 160, 80), (40, 25), CLINICAL, nmat=3, nvec=16),
        # Fewer candidates than a full block of vectors, half-precision values.
        _case("batched_2x5_f16", "batched", "f16", (131, 117, 61), (27, 23), CLINICAL, nmat=2, nvec=5),
        # The paper's Half/double configuration: half values, double vectors.
        _case("half_double_mid", "dose64", "f16", (200, 200, 120), (50, 50), CLINICAL),
        # Robust objective of a three-beam plan over three setup shifts, expected value
        # (half the width of the three-beam plan's grid and lattice).
        _case("robust_3x3", "robust", "u16", (80, 80, 50), (20, 13), CLINICAL, nmat=3, mode="expected"),
        # FP32 values with compensated sums on long rows, for reference doses.
        _case("dose_compensated_f32", "dose", "f32", (171, 155, 91), (41, 31), CLINICAL, compensated=True),
        # Tens of thousands of spots a quarter voxel apart, rows of up to thousands
        # of entries (a few slices of the beam shaped like the paper's liver beam 1).
        _case("dose_wide", "dose", "u16", (150, 150, 6), (272, 250), LIVER),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["dose", "dose", "objective", "objective", "autograd", "batched", "dose64", "pg", "robust", "wide"])
    if op == "wide":  # many close spots: rows of hundreds to thousands of entries
        sp = rng.uniform(0.25, 0.5)
        sx, sy = rng.randint(130, 272), rng.randint(130, 250)
        return _case("", rng.choice(["dose", "dose64"]), rng.choice(["u16", "f16"]),
                     (rng.randint(100, 150), rng.randint(100, 150), rng.randint(2, 5)), (sx, sy),
                     dict(dx=sp, dy=sp, sigma=4.0, tau=0.028798))
    if op == "pg":
        return _case("", op, rng.choice(["u16", "bf16"]), (rng.randint(24, 64), rng.randint(24, 64), rng.randint(12, 32)),
                     (rng.randint(15, 30), rng.randint(12, 24)), TINY, iters=rng.randint(10, 100))
    if op == "robust":
        return _case("", op, "u16", (rng.randint(40, 80), rng.randint(40, 80), rng.randint(30, 50)),
                     (rng.randint(10, 24), rng.randint(8, 15)), CLINICAL, nmat=rng.randint(2, 3),
                     mode=rng.choice(["expected", "worst"]))
    nx = _log_int(rng, 48, 230)
    ny = max(32, min(230, int(nx * rng.uniform(0.75, 1.25))))
    nz = _log_int(rng, 24, 120)
    fill = rng.uniform(0.2, 0.4)  # share of the lateral width that the spots cover
    sx, sy = max(8, int(nx * fill / 1.25)), max(8, int(ny * fill / 1.25))
    fmt = rng.choice(["u16", "u16", "bf16", "f16", "fp8", "f32"])
    more = {}
    if op == "dose":
        more = rng.choice([{}, {}, {"compensated": True}, {"index16": True}])
    elif op == "dose64":
        fmt = rng.choice(["f16", "f16", "u16", "bf16"])
    elif op == "batched":
        fmt = rng.choice(["u16", "u16", "bf16", "fp8"])
        nx, ny, nz = min(nx, 160), min(ny, 160), min(nz, 80)
        more = dict(nmat=rng.randint(1, 3), nvec=rng.randint(1, 16))
    model = dict(dx=1.25, dy=1.25, sigma=rng.uniform(3.0, 4.0), tau=0.009134)
    return _case("", op, fmt, (nx, ny, nz), (sx, sy), model, **more)


# ---------------------------------------------------------------- matrices

SHIFTS = [(0.0, 0.0), (-3.0, 3.0), (3.0, 0.0), (0.0, -3.0), (-3.0, -3.0), (3.0, 3.0), (-3.0, 0.0), (0.0, 3.0), (3.0, -3.0)]


def _uniform(n, seed, dtype=torch.float32):
    g = torch.Generator()
    g.manual_seed(seed)
    return torch.rand(n, generator=g, dtype=dtype).cuda()


def _beam(c, seed, shift=(0.0, 0.0), grid=None):
    """Row pointers (int64), columns (int32, ascending in a row) and values (FP32)
    of one pencil beam along +z on the GPU; row (iz * ny + iy) * nx + ix."""
    nx, ny, nz = grid or (c["nx"], c["ny"], c["nz"])
    sx, sy, dx, dy, sigma, tau = c["sx"], c["sy"], c["dx"], c["dy"], c["sigma"], c["tau"]
    dev = "cuda"
    depth = nz * (0.4 + 0.4 * _uniform(sx * sy, seed))             # Bragg depth of each spot
    z = torch.arange(nz, device=dev) + 0.5
    t = z[:, None] / depth[None, :]
    curve = torch.where(t <= 1.0, 0.3 + 0.7 * t ** 4, torch.exp(-0.5 * (z[:, None] - depth[None, :]) ** 2))
    r2 = -2.0 * sigma * sigma * math.log(tau)
    r = math.sqrt(r2)

    def axis(n, s, d, sh):  # candidate spots of each voxel coordinate and their offsets
        first = 0.5 * n - 0.5 * (s - 1) * d + sh
        v = torch.arange(n, device=dev) + 0.5
        a = torch.ceil((v - r - first) / d)[:, None] + torch.arange(int(2 * r / d) + 2, device=dev)
        return a.to(torch.int32), v[:, None] - (first + a * d), (a >= 0) & (a < s)

    ax, ex, okx = axis(nx, sx, dx, shift[0])
    ay, ey, oky = axis(ny, sy, dy, shift[1])
    live = (oky.any(1)[:, None] & okx.any(1)[None, :]).reshape(-1).nonzero()[:, 0]
    iy, ix = live // nx, live % nx
    rho2 = ey[iy][:, :, None] ** 2 + ex[ix][:, None, :] ** 2
    g = torch.where(oky[iy][:, :, None] & okx[ix][:, None, :] & (rho2 <= r2), torch.exp(rho2 / (-2.0 * sigma * sigma)), 0.0)
    cand = (ay[iy][:, :, None] * sx + ax[ix][:, None, :]).clamp_(0, sx * sy - 1)
    g, cand = g.reshape(live.numel(), -1), cand.reshape(live.numel(), -1)
    del rho2
    cnt = torch.zeros(nz, ny * nx, dtype=torch.int64, device=dev)
    cols, vals = [], []
    for iz in range(nz):
        v = g * curve[iz][cand]
        m = v >= tau
        cnt[iz, live] = m.sum(1)
        cols.append(cand[m])
        vals.append(v[m])
    rp = torch.zeros(nz * ny * nx + 1, dtype=torch.int64, device=dev)
    torch.cumsum(cnt.reshape(-1), 0, out=rp[1:])
    return rp, torch.cat(cols), torch.cat(vals)


def _rows(rp):
    return torch.repeat_interleave(torch.arange(rp.numel() - 1, device=rp.device), rp[1:] - rp[:-1])


def _encode(fmt, rp, v, top=None):
    """(codes, scales, decoded FP64 values) of FP32 values in a stored format."""
    if fmt == "u16":
        s = (v.max() if top is None else top) / 65535.0
        q = torch.round(v / s).clamp_(0, 65535).to(torch.int32)
        return q.to(torch.int16), s.reshape(1).float(), lambda: q.double() * s.double()
    if fmt == "fp8":
        rows = _rows(rp)
        top = torch.zeros(rp.numel() - 1, device=v.device).scatter_reduce_(0, rows, v, "amax")
        s = torch.where(top > 0, top / 448.0, 1.0)
        q = (v / s[rows]).clamp_(max=448.0).to(torch.float8_e4m3fn)
        return q.view(torch.uint8), s, lambda: q.float().double() * s.double()[rows]
    q = v.to({"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}[fmt])
    return q.view(VALUE_DTYPE[fmt]), None, lambda: q.double()


def _along(c, seed, shift, axis):
    """A beam entering the patient grid along +z, +x or +y: generated with that
    axis as depth, rows put in patient voxel order."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if axis == "z":
        return _beam(c, seed, shift)
    gx, gy, gz = (ny, nz, nx) if axis == "x" else (nz, nx, ny)
    rp, col, val = _beam(c, seed, shift, (gx, gy, gz))
    src = torch.arange(nx * ny * nz, device="cuda").reshape(gz, gy, gx)  # [depth][second][first]
    src = (src.permute(1, 2, 0) if axis == "x" else src.permute(2, 0, 1)).reshape(-1)  # patient [z][y][x]
    lens = (rp[1:] - rp[:-1])[src]
    out = torch.zeros_like(rp)
    torch.cumsum(lens, 0, out=out[1:])
    take = torch.repeat_interleave(rp[src] - out[:-1], lens) + torch.arange(col.numel(), device="cuda")
    return out, col[take], val[take]


def _matrices(c, seed):
    """The case's matrices: (row pointers, columns, values FP32, columns' count) each; a
    robust plan gives one such list of beams per scenario."""
    n = c["sx"] * c["sy"]
    if c["op"] == "robust":
        return [[(*_along(c, 1000 * seed + 7 + b, SHIFTS[s], "zxy"[b]), n) for b in range(3)] for s in range(c["nmat"])]
    return [(*_beam(c, 1000 * seed + 1, SHIFTS[s]), n) for s in range(c.get("nmat", 1))]


def _target(c):
    """Prescription and weights: an ellipsoid around the grid centre at 0.6 of the depth."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    ax = [(torch.arange(n, device="cuda") + 0.5 - f * n) / (0.12 * n) for n, f in ((nx, 0.5), (ny, 0.5), (nz, 0.6))]
    inside = (ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2 <= 1.0).reshape(-1)
    return torch.where(inside, 60.0, 0.0), torch.where(inside, 10.0, 1.0)


def _vectors(c, seed, ncols):
    op, nrows = c["op"], c["nx"] * c["ny"] * c["nz"]
    v = {}
    if op == "batched":
        v["X"] = [_uniform(ncols * c["nvec"], 500 * seed + 3 + i).reshape(ncols, c["nvec"]) for i in range(c["nmat"])]
    elif op == "dose64":
        v["x"] = _uniform(ncols, 500 * seed + 3, torch.float64)
    else:
        v["x"] = _uniform(ncols, 500 * seed + 3)
    if op in ("objective", "robust", "pg"):
        v["p"], v["w"] = _target(c)
    if op == "autograd":  # the residual of a caller's objective: mixed signs
        v["r"] = _uniform(nrows, 500 * seed + 9) - 0.5
    return v


def _eta(c):
    """Step size of the projected-gradient loop: below 1 / (2 max w |A|_1 |A|_inf) of
    these beams, a row and a column summing to at most their Gaussian's mass."""
    mass = 2.0 * math.pi * c["sigma"] ** 2
    return 1.0 / (2.0 * 10.0 * (mass / (c["dx"] * c["dy"])) * (mass * c["nz"]))


# ---------------------------------------------------------------- the cases

def prepare(case, seed):
    c, st = case, {"op": case["op"], "case": case}
    mats = _matrices(c, seed)
    if c["op"] == "robust":
        top = torch.stack([m[2].max() for beams in mats for m in beams]).max()
        handles = []
        for beams in mats:
            host = []
            for rp, col, val, n in beams:
                q, s, _ = _encode("u16", rp, val, top)
                host.append((rp.cpu().numpy().astype(np.uint32), col.cpu().numpy().view(np.uint32), n,
                             q.cpu().numpy().view(np.uint16), s.cpu().numpy()))
            handles.append(dose.DoseMatrix.from_multibeam(host, fmt="u16"))
        st["set"] = dose.ScenarioSet(handles)
        st["f_scen"] = torch.empty(len(handles), dtype=torch.float64, device="cuda")
    else:
        handles = []
        for rp, col, val, n in mats:
            q, s, _ = _encode(c["fmt"], rp, val)
            handles.append(dose.DoseMatrix.from_csr(rp.to(torch.int32), col, ncols=n, fmt=c["fmt"], values=q, scales=s,
                                                    compensated=c.get("compensated", False),
                                                    index16=c.get("index16", False)))
    del mats
    st["A"] = handles
    st.update(_vectors(c, seed, handles[0].ncols))
    if c["op"] == "autograd":
        st["x"].requires_grad_(True)
    if c["op"] == "pg":
        st["x0"] = st["x"].clone()
        st["solver"] = dose.PGSolver(handles[0], st["x"], st["p"], st["w"], _eta(c), c["iters"])
    torch.cuda.synchronize()
    return st


def run(st):
    op, A = st["op"], st["A"]
    if op == "dose":
        return A[0].spmv(st["x"])
    if op == "dose64":
        return A[0].spmv_f64(st["x"])
    if op == "objective":
        f, g, d = A[0].fwd_adj_quadratic(st["x"], st["p"], st["w"], want_d=True)
        return {"f": f, "g": g, "d": d}
    if op == "autograd":
        d = dose.dose_spmv(A[0], st["x"])
        (g,) = torch.autograd.grad(d, st["x"], st["r"])
        return {"d": d.detach(), "g": g}
    if op == "batched":
        return dose.spmv_batched(A, st["X"])
    if op == "robust":
        f, g, fs = st["set"].robust_quadratic(st["x"], st["p"], st["w"], mode=st["case"]["mode"], f_scen=st["f_scen"])
        return {"f": f, "g": g, "f_scen": fs}
    st["x"].copy_(st["x0"])  # every pass starts the same optimisation
    return {"f": st["solver"].run(), "x": st["x"]}


def _entries(c):
    """Expected entries of one matrix: each spot's disc of voxels above the
    threshold, slice by slice, clipped to the grid (Bragg depths at their quantiles)."""
    total = 0.0
    for b, (nx, ny, nz) in enumerate([(c["nx"], c["ny"], c["nz"]), (c["ny"], c["nz"], c["nx"]), (c["nz"], c["nx"], c["ny"])]):
        if b and c["op"] != "robust":
            break
        z = np.arange(nz)[:, None] + 0.5
        zj = nz * (0.4 + 0.4 * (np.arange(32) + 0.5) / 32)
        t = z / zj
        curve = np.where(t <= 1, 0.3 + 0.7 * t ** 4, np.exp(-0.5 * (z - zj) ** 2))
        r = np.sqrt(np.maximum(0.0, 2 * c["sigma"] ** 2 * np.log(np.maximum(curve / c["tau"], 1e-30))))

        def share(n, s, d):  # mean share of a disc's width (about 1.7 r across) inside the grid
            x0 = 0.5 * n - 0.5 * (s - 1) * d + d * np.arange(s)[:, None]
            h = 0.85 * r.reshape(1, -1) + 1e-9
            return (np.clip(x0 + h, 0, n) - np.clip(x0 - h, 0, n)).mean(0) / (2 * h[0])

        inside = share(nx, c["sx"], c["dx"]) * share(ny, c["sy"], c["dy"])
        total += c["sx"] * c["sy"] * float((math.pi * r.reshape(-1) ** 2 * inside).sum()) / 32
    return total


def work(case):
    """Bytes: every entry's stored value once (their columns follow from the
    lattice and could be coded in next to nothing), the vectors once."""
    c, op = case, case["op"]
    nrows, ncols, nnz = c["nx"] * c["ny"] * c["nz"], c["sx"] * c["sy"], _entries(c)
    k, nmat = c.get("nvec", 1), c.get("nmat", 1)
    a = nnz * VALUE_BYTES[c["fmt"]] + (4 * nrows if c["fmt"] == "fp8" else 0)
    if op == "dose":
        return {"bytes": a + 4 * (nrows + ncols), "flops": 2 * nnz}
    if op == "dose64":
        return {"bytes": a + 8 * (nrows + ncols), "flops": 2 * nnz}
    if op == "objective":
        return {"bytes": a + 12 * nrows + 8 * ncols, "flops": 4 * nnz + 5 * nrows}
    if op == "autograd":  # two passes: the residual comes between them
        return {"bytes": 2 * a + 8 * nrows + 8 * ncols, "flops": 4 * nnz}
    if op == "batched":
        return {"bytes": nmat * (a + 4 * k * (nrows + ncols)), "flops": nmat * 2 * k * nnz}
    if op == "robust":
        return {"bytes": nmat * a + 8 * nrows + 8 * 3 * ncols, "flops": nmat * (4 * nnz + 5 * nrows)}
    n = c["iters"]  # a small matrix stays on the chip: it and the vectors are read once
    return {"bytes": a + 8 * nrows + 8 * ncols, "flops": n * (4 * nnz + 5 * nrows)}


def _forward(rows, col, a, x, nrows):
    y = torch.zeros((nrows,) + tuple(x.shape[1:]), dtype=torch.float64, device="cuda")
    if x.dim() == 2:  # one vector at a time: the products of all would not fit
        for j in range(x.shape[1]):
            y[:, j] = _forward(rows, col, a, x[:, j], nrows)
        return y
    return y.index_add_(0, rows, a * x[col])


def exact(case, seed):
    c, op = case, case["op"]
    nrows = c["nx"] * c["ny"] * c["nz"]
    mats = _matrices(c, seed)
    if op == "robust":
        top = torch.stack([m[2].max() for beams in mats for m in beams]).max()
        parts = [[(_rows(rp), col.long() + b * n, _encode("u16", rp, val, top)[2]()) for b, (rp, col, val, n) in
                  enumerate(beams)] for beams in mats]
        mats = [[torch.cat([p[i] for p in beams]) for i in range(3)] for beams in parts]
        ncols = 3 * c["sx"] * c["sy"]
    else:
        mats = [[_rows(rp), col.long(), _encode(c["fmt"], rp, val)[2]()] for rp, col, val, _ in mats]
        ncols = c["sx"] * c["sy"]
    v = _vectors(c, seed, ncols)
    if op == "batched":
        return [_forward(*m, X.double(), nrows) for m, X in zip(mats, v["X"])]
    rows, col, a = mats[0]
    x = v["x"].double()
    if op in ("dose", "dose64"):
        return _forward(rows, col, a, x, nrows)

    def back(rows, col, a, r):
        return torch.zeros(ncols, dtype=torch.float64, device="cuda").index_add_(0, col, a * r[rows])

    if op == "autograd":
        return {"d": _forward(rows, col, a, x, nrows), "g": back(rows, col, a, v["r"].double())}
    p, w = v["p"].double(), v["w"].double()

    def objective(rows, col, a, x):
        d = _forward(rows, col, a, x, nrows)
        return (w * (d - p) ** 2).sum().reshape(1), back(rows, col, a, 2 * w * (d - p)), d

    if op == "objective":
        f, g, d = objective(rows, col, a, x)
        return {"f": f, "g": g, "d": d}
    if op == "robust":
        got = [objective(*m, x) for m in mats]
        fs = torch.cat([t[0] for t in got])
        if c["mode"] == "worst":
            return {"f": fs.max().reshape(1), "g": got[int(fs.argmax())][1], "f_scen": fs}
        return {"f": fs.mean().reshape(1), "g": torch.stack([t[1] for t in got]).mean(0), "f_scen": fs}
    eta = float(np.float32(_eta(c)))
    hist = []
    for _ in range(c["iters"]):
        f, g, _ = objective(rows, col, a, x)
        hist.append(f)
        x = (x - eta * g).clamp_(min=0)
    return {"f": torch.cat(hist), "x": x}
