"""Timed cases of the library: what a proton-CT reconstruction program has it do.

Every case is a dict of plain values with a "kind":

  cycles       NTVS cycles on a loaded system (the reconstruction itself): set the image, run
               K cycles (N TV steps and one block-DROP sweep each), read the image
  paths        the same with the rows traced from path records in every sweep
  batch        K cycles of many uneven reconstructions advanced together, images read back
  project      the forward projection A x of a loaded system
  initial      the initial iterate: binning, Ram-Lak, back-projection, median, hull
  reconstruct  the whole program from a device-resident CSR system: load, K cycles, read-back

Sizes are those of the synthetic workloads the benchmark and the tests use (32x32x1 slice,
scaled 3D phantoms, 200x200x16 CTP404, 256x256x64 traced rows, sweep members of 64..128
voxels a side), at their history counts or a fraction of them.  Relaxations are the
workloads' 1e-4..1e-3, or 0.3, at which a sweep's update is large in an FP32 image.

Inputs are made on the GPU from the seed: a cylinder phantom with inserts, bent or straight
histories over a full turn, WEPL with 1 % noise, and an initial image with the noise of a
filtered back-projection.  "binned" rows are ordered by slice and lateral offset inside an
angle, "listmode" rows come as detected, in random order inside an angle.
"""
import math

import numpy as np
import torch

import paper_1803_01112_gb300 as ntvs

DEV = "cuda"
ALPHA = 0.75
_VAL = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_RSP = (0.0013, 0.0013, 0.877, 0.9973, 1.0386, 1.155, 1.356, 1.8)   # the phantom's inserts
_MIN_LEN = 1e-4


def _system(name, kind, nx, ny, nz, hist, angles, blocks, N, K, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, dx=1.0, dz=2.5, hist=hist, angles=angles, curved=True,
             order="binned", blocks=blocks, val="f32", compute="f32", storage="csr32", N=N, K=K, lam=2e-4,
             check=False, rule="ntvs")
    c.update(kw)
    return c


def listed():
    return [
        # the smallest use: one 2D slice in FP64, where launches and latency are the time
        _system("slice32_f64", "cycles", 32, 32, 1, 20_000, 90, 10, 3, 4, curved=False, val="f64", compute="f64",
                lam=1e-3),
        # a small 3D volume with odd sizes and ragged blocks, FP32: a scanner's quick preview
        _system("preview_f32", "cycles", 41, 37, 5, 40_003, 60, 7, 3, 4, lam=0.3),
        # a mid-sized object with the TV-reduction check on and six steps per cycle
        _system("object128_check_f32", "cycles", 128, 128, 16, 800_000, 90, 20, 6, 1, check=True),
        # the full CTP404 scan, one cycle, FP32: the headline workload
        _system("ctp404_f32", "cycles", 200, 200, 16, 10_000_000, 360, 20, 3, 1),
        # the same geometry with BF16 lengths and packed 16-bit column offsets
        _system("ctp404_bf16_delta16", "cycles", 200, 200, 16, 2_000_000, 360, 20, 3, 1, val="bf16",
                storage="delta16", lam=0.3),
        # FP64 values and arithmetic at the full grid: the reference-quality run
        _system("ctp404_f64", "cycles", 200, 200, 16, 500_000, 360, 20, 3, 1, val="f64", compute="f64",
                lam=0.3),
        # histories in the order they were detected (no binning by slice)
        _system("ctp404_listmode_f32", "cycles", 200, 200, 16, 2_000_000, 360, 20, 3, 1, order="listmode",
                lam=0.3),
        # rows traced on the fly on the large grid
        dict(name="traced_256", kind="paths", nx=256, ny=256, nz=64, dx=0.8, dz=1.25, hist=4_000_000, angles=720,
             curved=True, order="binned", blocks=40, N=4, K=1, lam=0.3, n_seg=16),
        # a parameter sweep: uneven members advanced together
        dict(name="sweep_16", kind="batch", members=16, side_lo=64, side_hi=128, nz_lo=8, nz_hi=16, hist_lo=100_000,
             hist_hi=500_000, blocks=20, K=2, angles=90),
        # A x of a loaded system: simulating the data, or the residual of every history
        _system("project_f32", "project", 200, 200, 16, 2_000_000, 360, 20, 3, 1),
        # the initial image of a full scan
        dict(name="initial_10M", kind="initial", nx=200, ny=200, nz=16, dx=1.0, dz=2.5, hist=10_000_000, angles=360,
             curved=False, order="binned", n_theta=180, n_t=160, radius=2, ball=False, tau=0.3),
        # the whole program on a new system: load, twelve cycles, read the image
        _system("reconstruct_96", "reconstruct", 96, 96, 12, 500_000, 90, 20, 3, 12),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["cycles", "cycles", "cycles", "cycles", "paths", "batch", "project", "initial", "reconstruct"])
    nx, ny, nz = logint(24, 200), logint(24, 200), rng.randint(1, 16)
    hist = logint(15_000, 2_000_000)
    if kind == "batch":
        lo = rng.randint(4, 10) * 8
        return dict(kind=kind, members=rng.randint(3, 20), side_lo=lo, side_hi=lo + rng.randint(1, 6) * 8,
                    nz_lo=rng.randint(2, 8), nz_hi=rng.randint(9, 16), hist_lo=logint(5_000, 40_000),
                    hist_hi=logint(50_000, 400_000), blocks=rng.randint(4, 20), K=rng.randint(1, 3), angles=90)
    if kind == "paths":
        return dict(kind=kind, nx=logint(48, 256), ny=logint(48, 256), nz=rng.randint(4, 64), dx=0.8, dz=1.25,
                    hist=hist, angles=rng.choice([90, 360, 720]), curved=rng.random() < 0.8,
                    order=rng.choice(["binned", "binned", "listmode"]), blocks=rng.randint(5, 40), N=rng.randint(1, 6),
                    K=1, lam=rng.choice([1e-4, 2e-4, 5e-4]), n_seg=rng.choice([8, 16, 16, 24]))
    if kind == "initial":
        angles = rng.choice([90, 360])   # every projection on the centre of an angle bin
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, dx=1.0, dz=2.5, hist=logint(50_000, 10_000_000),
                    angles=angles, curved=False, order=rng.choice(["binned", "listmode"]),
                    n_theta=180 if angles == 360 else rng.choice([90, 180]), n_t=logint(32, 200), radius=rng.choice([1, 2, 2, 3]),
                    ball=rng.random() < 0.25, tau=rng.choice([0.2, 0.3]))
    val = rng.choice(["f32", "f32", "f32", "f64", "bf16", "f16"])
    c = _system("", kind, nx, ny, nz, hist, rng.choice([60, 90, 360]), rng.randint(3, 24), rng.randint(1, 6),
                12 if kind == "reconstruct" else rng.randint(1, 2), val=val,
                compute="f64" if val == "f64" or (val == "f32" and rng.random() < 0.15) else "f32",
                storage="delta16" if val in ("bf16", "f16") and rng.random() < 0.6 else "csr32",
                order=rng.choice(["binned", "binned", "listmode"]), curved=rng.random() < 0.8,
                lam=rng.choice([1e-4, 2e-4, 5e-4, 0.3]), check=rng.random() < 0.3)
    if not c["check"]:
        c["rule"] = rng.choice(["ntvs", "ntvs", "ntvs", "decoupled"])
    if c["compute"] == "f64":
        c["hist"] = min(hist, 500_000)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, n, lo=0.0, hi=1.0, dtype=torch.float32):
    return torch.rand(n, generator=g, device=DEV, dtype=dtype) * (hi - lo) + lo


def _cylinders(c):
    """[(cx, cy, r, rsp difference)] of the phantom: a cylinder and eight inserts."""
    R = 0.375 * min(c["nx"], c["ny"]) * c["dx"]
    ins = [(0.8 * R * math.cos(math.pi * q / 4), 0.8 * R * math.sin(math.pi * q / 4), 0.08 * R, v - 1.0)
           for q, v in enumerate(_RSP)]
    return [(0.0, 0.0, R, 1.0)] + ins


def _phantom(c):
    x = (torch.arange(c["nx"], device=DEV, dtype=torch.float64) + 0.5 - 0.5 * c["nx"]) * c["dx"]
    y = (torch.arange(c["ny"], device=DEV, dtype=torch.float64) + 0.5 - 0.5 * c["ny"]) * c["dx"]
    img = torch.zeros(c["ny"], c["nx"], device=DEV, dtype=torch.float64)
    for cx, cy, r, v in _cylinders(c):
        img += v * (((x[None, :] - cx) ** 2 + (y[:, None] - cy) ** 2) <= r * r)
    return img[None].expand(c["nz"], -1, -1).reshape(-1)


def _image(c, seed):
    """The phantom with the noise of a back-projection."""
    V = c["nx"] * c["ny"] * c["nz"]
    return _phantom(c) + 0.02 * torch.randn(V, generator=_gen(seed + 77), device=DEV, dtype=torch.float64)


def _paths(c, seed):
    """(path records float32 [M, 10], WEPL noise factors float64 [M]) in acquisition order."""
    g = _gen(seed)
    M, A, nz, dz = c["hist"], c["angles"], c["nz"], c["dz"]
    a = torch.arange(M, device=DEV) * A // M                                 # angle by angle
    R = 0.375 * min(c["nx"], c["ny"]) * c["dx"]
    t = _uniform(g, M, -R, R)
    z = _uniform(g, M, 0.0, nz * dz)
    if c["order"] == "binned":   # by slice, then by lateral offset, inside each angle
        key = (a * nz + (z / dz).long().clamp_(0, nz - 1)).double() + (t.double() + R) / (2.001 * R)
        p = torch.argsort(key)
        t, z = t[p], z[p]
        del key, p
    th = a.double() * (2.0 * math.pi / A)
    ux, uy = torch.cos(th).float(), torch.sin(th).float()
    del a, th
    px, py = -t * uy, t * ux
    hx, hy = 0.5 * c["nx"] * c["dx"], 0.5 * c["ny"] * c["dx"]
    lo = torch.full_like(t, -1e9)
    hi = torch.full_like(t, 1e9)
    for p, u, h in ((px, ux, hx), (py, uy, hy)):   # the line inside the grid square, 1 mm more at both ends
        s0, s1 = (-h - p) / u, (h - p) / u
        ok = u.abs() > 1e-6
        lo = torch.where(ok, torch.maximum(lo, torch.minimum(s0, s1)), lo)
        hi = torch.where(ok, torch.minimum(hi, torch.maximum(s0, s1)), hi)
    lo, hi = lo - 1.0, hi + 1.0
    rec = torch.zeros(M, 10, device=DEV, dtype=torch.float32)
    rec[:, 0], rec[:, 1], rec[:, 2] = px + lo * ux, py + lo * uy, z
    rec[:, 3], rec[:, 4], rec[:, 5] = px + hi * ux, py + hi * uy, z
    if c["curved"]:   # cubic bends of at most about 2 mm, sideways and along z
        k = 27.0 / 8.0 * min(2.0, 4.0 * c["nx"] / 200.0)
        for q in range(6, 10):
            rec[:, q] = _uniform(g, M, -k, k)
    return rec, 1.0 + 0.01 * torch.randn(M, generator=g, device=DEV, dtype=torch.float64)


def _chord_wepl(c, rec):
    """WEPL of the straight chords through the phantom's cylinders."""
    P, Q = rec[:, 0:2].double(), rec[:, 3:5].double()
    u = (Q - P) / (Q - P).norm(dim=1, keepdim=True)
    w = torch.zeros(rec.shape[0], device=DEV, dtype=torch.float64)
    for cx, cy, r, v in _cylinders(c):
        d = (P[:, 0] - cx) * u[:, 1] - (P[:, 1] - cy) * u[:, 0]
        w += 2.0 * v * torch.sqrt(torch.clamp(r * r - d * d, min=0.0))
    return w


def _row_wepl(x, n, vox, ln):
    """Line integrals of the image x along traced rows of n entries each."""
    row = torch.repeat_interleave(torch.arange(n.numel(), device=DEV), n)
    return torch.zeros(n.numel(), device=DEV, dtype=torch.float64).index_add_(0, row, ln.double() * x[vox.long()])


def _path_wepl(c, rec, n_seg):
    x = _phantom(c)
    return torch.cat([_row_wepl(x, n, v, ln) for _, n, v, ln in _trace(c, rec, n_seg, torch.float32)])


def _trace(c, rec, n_seg, dt):
    """CSR rows of the path records: every straight segment cut at the voxel planes it
    crosses, consecutive pieces of one voxel merged, short ones dropped.  Yields
    (first row, entries per row, columns int32, lengths) for runs of rows."""
    M = rec.shape[0]
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    step = max(1, 40_000_000 // (nx + ny + nz + 4 * n_seg))
    org = (-0.5 * nx * c["dx"], -0.5 * ny * c["dx"], 0.0)
    size = (c["dx"], c["dx"], c["dz"])
    s = torch.linspace(0, 1, n_seg + 1, device=DEV, dtype=dt)
    h10, h11 = s ** 3 - 2 * s ** 2 + s, s ** 3 - s ** 2
    for r0 in range(0, M, step):
        p = rec[r0:r0 + step].to(dt)
        m = p.shape[0]
        ch = p[:, 3:5] - p[:, 0:2]
        u = ch / ch.norm(dim=1, keepdim=True)
        ol = p[:, 6:7] * h10 + p[:, 7:8] * h11
        oz = p[:, 8:9] * h10 + p[:, 9:10] * h11
        pts = [p[:, 0:1] + s * (p[:, 3:4] - p[:, 0:1]) - ol * u[:, 1:2],
               p[:, 1:2] + s * (p[:, 4:5] - p[:, 1:2]) + ol * u[:, 0:1],
               p[:, 2:3] + s * (p[:, 5:6] - p[:, 2:3]) + oz]
        P = [q[:, :-1].reshape(-1, 1) for q in pts]
        D = [(q[:, 1:] - q[:, :-1]).reshape(-1, 1) for q in pts]
        one = torch.ones_like(P[0])
        cuts = [torch.zeros_like(one)]
        for q in range(3):
            n = int(torch.ceil((D[q].abs() / size[q]).max()).item()) + 1
            k = torch.ceil((torch.minimum(P[q], P[q] + D[q]) - org[q]) / size[q])
            k = k + torch.arange(n, device=DEV, dtype=dt)
            t = (org[q] + k * size[q] - P[q]) / D[q]
            cuts.append(torch.where((t > 0) & (t < 1), t, one))
            del k, t
        T = torch.sort(torch.cat(cuts + [one], dim=1), dim=1).values
        del cuts
        ln = T[:, 1:] - T[:, :-1]
        mid = T[:, :-1] + 0.5 * ln
        del T
        ln *= torch.sqrt(D[0] ** 2 + D[1] ** 2 + D[2] ** 2)
        keep = ln > 1e-6
        vox = torch.zeros(ln.shape, device=DEV, dtype=torch.int32)
        for q, n in ((2, nz), (1, ny), (0, nx)):
            i = torch.floor((P[q] + mid * D[q] - org[q]) / size[q]).int()
            keep &= (i >= 0) & (i < n)
            vox.mul_(n).add_(i)
            del i
        row = torch.arange(m, device=DEV, dtype=torch.int32).repeat_interleave(n_seg)[:, None].expand(ln.shape)
        vox, row, ln = vox[keep], row[keep], ln[keep]
        del keep, mid
        if vox.numel():
            new = torch.ones(vox.numel(), device=DEV, dtype=torch.bool)
            new[1:] = (vox[1:] != vox[:-1]) | (row[1:] != row[:-1])
            at = torch.cumsum(new, 0) - 1
            ln = torch.zeros(int(at[-1].item()) + 1, device=DEV, dtype=dt).index_add_(0, at, ln)
            vox, row = vox[new], row[new]
            keep = ln >= _MIN_LEN
            vox, row, ln = vox[keep], row[keep], ln[keep]
            del at, new, keep
        yield r0, torch.bincount(row, minlength=m), vox, ln
        del vox, row, ln


def _n_seg(c):
    return 16 if c["curved"] else 8


def _csr(c, seed):
    """(row_ptr, col, val, b) on the GPU in the case's storage type."""
    rec, noise = _paths(c, seed)
    vt = _VAL[c["val"]]
    dt = torch.float64 if c["val"] == "f64" else torch.float32
    x = _phantom(c)
    cnt, cols, vals, w = [], [], [], []
    for _, n, v, ln in _trace(c, rec, _n_seg(c), dt):
        cnt.append(n)
        w.append(_row_wepl(x, n, v, ln))
        cols.append(v)
        vals.append(ln.to(vt))
    rp = torch.zeros(c["hist"] + 1, device=DEV, dtype=torch.int64)
    torch.cumsum(torch.cat(cnt), 0, out=rp[1:])
    del rec, cnt
    col = torch.cat(cols)
    del cols
    val = torch.cat(vals)
    del vals
    return rp, col, val, (torch.cat(w) * noise).to(torch.float64 if c["val"] == "f64" else torch.float32)


def _params(c):
    return ntvs.Params(lam=c["lam"], N=c["N"], alpha=ALPHA, seed=7, tv_check=c.get("check", False),
                       step_rule=ntvs.NTVS_STEP_DECOUPLED if c.get("rule") == "decoupled" else ntvs.NTVS_STEP_NTVS)


def _shape(c):
    return c["nx"], c["ny"], c["nz"]


def _members(c, seed):
    """The sweep's members as cases of their own, with their seeds."""
    rng = np.random.default_rng(1234 + c["members"])   # sizes and parameters belong to the case
    out = []
    for q in range(c["members"]):
        n = int(rng.integers(c["side_lo"] // 8, c["side_hi"] // 8 + 1)) * 8
        m = dict(nx=n, ny=n, nz=int(rng.integers(c["nz_lo"], c["nz_hi"] + 1)), dx=1.0, dz=2.5,
                 hist=int(rng.integers(c["hist_lo"], c["hist_hi"] + 1)), angles=c["angles"], curved=True,
                 order="binned", blocks=c["blocks"], N=int(rng.integers(1, 7)), K=c["K"],
                 lam=float(rng.choice([1e-4, 2e-4, 5e-4])), check=q % 4 == 3, val="f32")
        out.append((m, seed * 1000 + q))
    return out


def _geom(c):
    return ntvs.fbp_geom(c["nx"], c["ny"], c["nz"], c["dx"], c["dx"], c["dz"], c["n_theta"], c["n_t"],
                         0.75 * min(c["nx"], c["ny"]) * c["dx"] / c["n_t"], theta0=-0.5 * math.pi / c["n_theta"])


# ------------------------------------------------------------------ preparation
def _loaded(c, csr):
    r = ntvs.Reconstructor(0, torch.cuda.current_stream().cuda_stream)
    r.set_compute_dtype(ntvs.NTVS_F64 if c["compute"] == "f64" else ntvs.NTVS_F32)
    r.load(_shape(c), *csr, n_blocks=c["blocks"],
           storage=ntvs.NTVS_DELTA16 if c["storage"] == "delta16" else ntvs.NTVS_CSR32)
    r.set_params(_params(c))
    return r


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        bt = ntvs.Batch(0)
        for m, s in _members(c, seed):
            rec, noise = _paths(m, s)
            b, x0 = (_path_wepl(m, rec, 16) * noise).float(), _image(m, s)
            torch.cuda.synchronize()   # the batch works on a stream of its own
            bt.add_paths(_shape(m), (m["dx"], m["dx"], m["dz"]), rec, b, m["blocks"], _params(m), x0)
        bt.finalize(max_cycles=1 << 17)
        return dict(c=c, bt=bt)
    if kind == "initial":
        rec, noise = _paths(c, seed)
        w = _chord_wepl(c, rec) * noise
        g = _geom(c)
        V = c["nx"] * c["ny"] * c["nz"]
        return dict(c=c, g=g, rec=rec, w=w, out=torch.empty(V, device=DEV, dtype=torch.float64),
                    ws=torch.empty(ntvs.ntvs_fbp_workspace_bytes(g), device=DEV, dtype=torch.uint8))
    if kind == "paths":
        rec, noise = _paths(c, seed)
        b = (_path_wepl(c, rec, c["n_seg"]) * noise).float()
        r = ntvs.Reconstructor(0, torch.cuda.current_stream().cuda_stream)
        r.load_paths(_shape(c), (c["dx"], c["dx"], c["dz"]), rec, b, n_blocks=c["blocks"], n_seg=c["n_seg"])
        r.set_params(_params(c))
        x0 = _image(c, seed)
        return dict(c=c, r=r, x0=x0, out=torch.empty_like(x0, dtype=torch.float32))
    csr = _csr(c, seed)
    x0 = _image(c, seed)
    od = torch.float64 if c["compute"] == "f64" else torch.float32
    if kind == "reconstruct":
        return dict(c=c, csr=csr, x0=x0)
    r = _loaded(c, csr)
    if kind == "project":
        return dict(c=c, r=r, x0=x0.to(od), out=torch.empty(c["hist"], device=DEV, dtype=od))
    return dict(c=c, r=r, x0=x0, out=torch.empty_like(x0, dtype=od))


# ------------------------------------------------------------------ one pass
def _cycles(r, x0, K):
    r.set_image(x0)
    r.set_state(0, 0)
    r.run(K)


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "batch":
        bt = state["bt"]
        bt.run(c["K"])
        return [bt.get_image(i, np.float32) for i in range(c["members"])]
    if kind == "initial":
        ntvs.ntvs_initial_iterate(state["g"], state["rec"], state["w"], state["out"], median_radius=c["radius"],
                                  median_ball=c["ball"], use_hull=True, tau=c["tau"], workspace=state["ws"],
                                  stream=torch.cuda.current_stream().cuda_stream)
        return state["out"]
    if kind == "project":
        return state["r"].forward_project(state["x0"], state["out"])
    if kind == "reconstruct":
        r = _loaded(c, state["csr"])
        _cycles(r, state["x0"], c["K"])
        img = r.get_image(np.float64 if c["compute"] == "f64" else np.float32)
        r.close()
        return img
    _cycles(state["r"], state["x0"], c["K"])
    ntvs.ntvs_get_image(state["r"].handle, state["out"])
    return state["out"]


# ------------------------------------------------------------------ work
def _entries(c):
    """Mean entries of a row: a chord across the grid square within the beam, in voxels."""
    side = 0.5 * (c["nx"] + c["ny"])
    return 1.27 * side * 1.05 + (0.0 if not c["curved"] else 4.0)


def _cycle_bytes(c, entry, real):
    V = c["nx"] * c["ny"] * c["nz"]
    # every entry and row (extent, right-hand side, norm) once; per TV step the image read and
    # written; per block 1/s read, the image read and written
    return c["K"] * (c["hist"] * (_entries(c) * entry + 8 + 2 * real) + V * (c["N"] * 16 + c["blocks"] * (16 + real)))


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        ws = [(m, m["hist"] * _entries(m)) for m, _ in _members(c, 0)]
        return dict(bytes=sum(_cycle_bytes(m, 8, 4) for m, _ in ws), flops=sum(4 * e * c["K"] for _, e in ws))
    V = c["nx"] * c["ny"] * c["nz"]
    if kind == "initial":
        S = c["nz"] * c["n_theta"] * c["n_t"]
        return dict(bytes=c["hist"] * 32 + S * 16 + V * 8,
                    flops=S * c["n_t"] + V * c["n_theta"] * 6)
    nnz = c["hist"] * _entries(c)
    if kind == "paths":
        m = dict(c, hist=0)
        return dict(bytes=c["K"] * c["hist"] * 48 + _cycle_bytes(m, 0, 4), flops=c["K"] * nnz * 16)
    vb = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[c["val"]]
    entry = vb + (2 if c["storage"] == "delta16" else 4)
    real = 8 if c["compute"] == "f64" else 4
    if kind == "project":
        return dict(bytes=nnz * entry + c["hist"] * (8 + real) + V * real, flops=2 * nnz)
    w = dict(bytes=_cycle_bytes(c, entry, real), flops=c["K"] * nnz * 4)
    if kind == "reconstruct":
        w["bytes"] += nnz * (4 + vb)
    return w


# ------------------------------------------------------------------ the same in 64 bits
def _splitmix(seed, n):
    mask = (1 << 64) - 1
    z = (seed + (n + 1) * 0x9E3779B97F4A7C15) & mask
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
    return z ^ (z >> 31)


def _diffs(x):
    d = [torch.zeros_like(x) for _ in range(3)]
    d[0][:, :, :-1] = x[:, :, 1:] - x[:, :, :-1]
    d[1][:, :-1] = x[:, 1:] - x[:, :-1]
    d[2][:-1] = x[1:] - x[:-1]
    return d


def _tv(x):
    d = _diffs(x)
    return torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2).sum()


def _tv_grad(x, eps):
    d = _diffs(x)
    D = torch.sqrt(eps + d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    q = [v / D for v in d]
    g = -(q[0] + q[1] + q[2])
    g[:, :, 1:] += q[0][:, :, :-1]
    g[:, 1:] += q[1][:, :-1]
    g[1:] += q[2][:-1]
    return g


def _runs(rp, r0, r1, most=40_000_000):
    """Row ranges of [r0, r1) of at most about `most` entries."""
    while r0 < r1:
        e = int(rp[r0].item()) + most
        q = int(torch.searchsorted(rp, e, right=True).item()) - 1
        q = min(r1, max(q, r0 + 1))
        yield r0, q
        r0 = q


def _part(csr, a, e):
    rp, col, val, b = csr
    e0, e1 = int(rp[a].item()), int(rp[e].item())
    row = torch.repeat_interleave(torch.arange(e - a, device=DEV), rp[a + 1:e + 1] - rp[a:e])
    return row, col[e0:e1].long(), val[e0:e1].double(), b[a:e].double()


def _ntvs_exact(c, csr, x0):
    prm = _params(c)
    shape = (c["nz"], c["ny"], c["nx"])
    x = x0.double().clone()
    rp, M, B = csr[0], c["hist"], c["blocks"]
    per = -(-M // B)
    ell_prev = 0
    for k in range(c["K"]):
        lo, hi = min(k, ell_prev), max(k, ell_prev)
        ell = lo + _splitmix(prm.seed, k) % (hi - lo + 1)
        for n in range(c["N"]):
            g = _tv_grad(x.view(shape), prm.eps_tv).reshape(-1)
            gn = float(torch.sqrt((g * g).sum()))
            phi = _tv(x.view(shape)) if prm.tv_check else None
            for _ in range(prm.max_retries):
                beta = prm.beta0 * prm.alpha ** ell
                if c.get("rule") == "decoupled":
                    beta = prm.beta0 * prm.alpha ** n * prm.gamma ** k
                z = x - (beta / gn) * g if gn > 0 else x
                ell += 1
                if not prm.tv_check or bool(_tv(z.view(shape)) <= phi):
                    x = z
                    break
        ell_prev = ell
        for t in range(B):
            r0, r1 = min(t * per, M), min((t + 1) * per, M)
            delta = torch.zeros_like(x)
            hits = torch.zeros(x.numel(), device=DEV, dtype=torch.int64)
            for a, e in _runs(rp, r0, r1):
                row, col, val, b = _part(csr, a, e)
                n2 = torch.zeros(e - a, device=DEV, dtype=torch.float64).index_add_(0, row, val * val)
                dot = torch.zeros(e - a, device=DEV, dtype=torch.float64).index_add_(0, row, val * x[col])
                res = torch.where(n2 > 0, (b - dot) / n2, torch.zeros_like(n2))
                delta.index_add_(0, col, val * res[row])
                hits += torch.bincount(col[val != 0], minlength=hits.numel())
                del row, col, val
            x = torch.where(hits > 0, x + prm.lam * delta / hits.clamp(min=1), x)
    return x


def _initial_exact(c, rec, w):
    g = _geom(c)
    nx, ny, nz, na, nt = c["nx"], c["ny"], c["nz"], c["n_theta"], c["n_t"]
    p = rec.double()
    ddx, ddy = p[:, 3] - p[:, 0], p[:, 4] - p[:, 1]
    ln = torch.sqrt(ddx * ddx + ddy * ddy)
    t = (p[:, 1] * ddx - p[:, 0] * ddy) / ln
    phi = torch.atan2(ddx, -ddy) - g.theta0
    turns = torch.floor(phi / math.pi)
    phi = phi - turns * math.pi
    t = torch.where(turns.long() % 2 != 0, -t, t)
    a = torch.floor(phi / (math.pi / na)).long().clamp(0, na - 1)
    u, v = t / g.dt + 0.5 * nt, 0.5 * (p[:, 2] + p[:, 5]) / g.dz
    ok = (u >= 0) & (u < nt) & (v >= 0) & (v < nz)
    key = ((v.long() * na + a) * nt + u.long())[ok]
    S = nz * na * nt
    cnt = torch.bincount(key, minlength=S)
    sino = torch.zeros(S, device=DEV, dtype=torch.float64).index_add_(0, key, w[ok])
    sino = torch.where(cnt > 0, sino / cnt.clamp(min=1), torch.zeros_like(sino)).view(nz, na, nt)
    m = torch.arange(nt, device=DEV, dtype=torch.float64)
    lag = m[:, None] - m[None, :]
    h = torch.where(lag.long() % 2 != 0, -1.0 / (math.pi ** 2 * lag * lag * g.dt ** 2), torch.zeros_like(lag))
    h = torch.where(lag == 0, torch.full_like(lag, 1.0 / (4.0 * g.dt ** 2)), h)
    q = g.dt * torch.matmul(sino, h)
    x = (torch.arange(nx, device=DEV, dtype=torch.float64) + 0.5 - 0.5 * nx) * g.dx
    y = (torch.arange(ny, device=DEV, dtype=torch.float64) + 0.5 - 0.5 * ny) * g.dy
    img = torch.zeros(nz, ny, nx, device=DEV, dtype=torch.float64)
    pad = torch.zeros(nz, na, nt + 2, device=DEV, dtype=torch.float64)
    pad[:, :, 1:-1] = q
    for i in range(na):
        th = g.theta0 + (i + 0.5) * math.pi / na
        uu = (x[None, :] * math.cos(th) + y[:, None] * math.sin(th)) / g.dt + 0.5 * nt - 0.5
        k = torch.floor(uu)
        f = uu - k
        inside = (k >= -1) & (k < nt)
        k = k.long().clamp(-1, nt - 1)
        img += torch.where(inside, (1 - f) * pad[:, i][:, k + 1] + f * pad[:, i][:, k + 2], torch.zeros_like(f))
    img *= math.pi / na
    r, rz = c["radius"], c["radius"] if c["ball"] else 0
    big = torch.full((nz + 2 * rz, ny + 2 * r, nx + 2 * r), math.inf, device=DEV, dtype=torch.float64)
    big[rz:rz + nz, r:r + ny, r:r + nx] = img
    win = [big[rz + oz:rz + oz + nz, r + oy:r + oy + ny, r + ox:r + ox + nx]
           for oz in range(-rz, rz + 1) for oy in range(-r, r + 1) for ox in range(-r, r + 1)
           if ox * ox + oy * oy + oz * oz <= r * r + 1]
    out = torch.empty_like(img)
    for iz in range(nz):
        s = torch.sort(torch.stack([v_[iz] for v_ in win]), dim=0).values
        n = torch.isfinite(s).sum(0, keepdim=True)
        out[iz] = torch.gather(s, 0, n // 2)[0]
    return torch.where(out <= c["tau"], torch.zeros_like(out), out).reshape(-1)


def _traced_csr(c, seed, n_seg):
    """The rows of path records in 64 bits."""
    rec, noise = _paths(c, seed)
    w = _path_wepl(c, rec, n_seg) * noise
    parts = [(n, v, ln) for _, n, v, ln in _trace(c, rec, n_seg, torch.float64)]
    rp = torch.zeros(c["hist"] + 1, device=DEV, dtype=torch.int64)
    torch.cumsum(torch.cat([p[0] for p in parts]), 0, out=rp[1:])
    return rp, torch.cat([p[1] for p in parts]), torch.cat([p[2] for p in parts]), w.float()


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        out = []
        for m, s in _members(c, seed):
            out.append(_ntvs_exact(m, _traced_csr(m, s, 16), _image(m, s)).cpu().numpy())
        return out
    if kind == "initial":
        rec, noise = _paths(c, seed)
        return _initial_exact(c, rec, _chord_wepl(c, rec) * noise)
    if kind == "paths":
        return _ntvs_exact(c, _traced_csr(c, seed, c["n_seg"]), _image(c, seed))
    csr = _csr(c, seed)
    if kind == "project":
        x = _image(c, seed)
        x = x if c["compute"] == "f64" else x.float().double()
        out = torch.zeros(c["hist"], device=DEV, dtype=torch.float64)
        for a, e in _runs(csr[0], 0, c["hist"]):
            row, col, val, _ = _part(csr, a, e)
            out[a:e].index_add_(0, row, val * x[col])
            del row, col, val
        return out
    x = _ntvs_exact(c, csr, _image(c, seed))
    return x.cpu().numpy() if kind == "reconstruct" else x
