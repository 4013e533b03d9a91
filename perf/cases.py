"""The work that users of this library have it do, as cases that can be timed and compared.

Every case is one call sequence on a resident context, as a reconstruction or planning program
makes it: the iterate set from device memory, a few superiorized iterations (`suppy_run`) or plain
sweeps (`suppy_sweep`) enqueued, the iterate read back into device memory.  The matrices are the
three workload families of the library (parallel-beam CT, straight-ray traveltime tomography,
pencil-beam radiotherapy) at the sizes of its benchmark, tests and serving mix, built here on the
GPU; images, noise, bounds and starting points come from the seed.  `exact` restates the iterations
in float64 with plain torch.
"""
import functools
import math

import numpy as np
import torch

import paper_2606_27086_gb300 as pk

DTYPES = {"f32": pk.SUPPY_F32, "bf16": pk.SUPPY_BF16, "f16": pk.SUPPY_F16}
MODES = {"cimmino": pk.SUPPY_CIMMINO, "bip": pk.SUPPY_BIP, "drop": pk.SUPPY_DROP,
         "el": pk.SUPPY_EL, "emr": pk.SUPPY_EMR}
OBJECTIVES = {"none": pk.SUPPY_OBJ_NONE, "tv": pk.SUPPY_OBJ_TV_ISO, "atv": pk.SUPPY_OBJ_TV_ANISO,
              "mean": pk.SUPPY_OBJ_LINEAR}
STRATEGIES = {"default": pk.STRATEGY_AUTO, "one_pass": pk.STRATEGY_ONE_PASS}


def _ct(name, H, W, angles, bins, iters, mode="cimmino", obj="tv", dtype="f32", strategy="default",
        blocks=1, call="run"):
    return dict(name=name, family="ct", H=H, W=W, angles=angles, bins=bins, iters=iters, mode=mode,
                obj=obj, dtype=dtype, strategy=strategy, blocks=blocks, call=call, nrhs=1)


def _seismic(name, H, W, sources, receivers, iters, nrhs=1, mode="cimmino", strategy="default", obj="tv"):
    return dict(name=name, family="seismic", H=H, W=W, sources=sources, receivers=receivers,
                iters=iters, mode=mode, obj=obj, dtype="f32", strategy=strategy, blocks=1,
                call="run", nrhs=nrhs)


def _rt(name, nx, ny, nz, ns, nzb, iters, mode="bip", split=False):
    return dict(name=name, family="rt", nx=nx, ny=ny, nz=nz, beams=9, ns=ns, nzb=nzb, iters=iters,
                mode=mode, obj="mean", dtype="f32", strategy="default", blocks=3, call="run",
                nrhs=1, split=split)


def listed():
    return [
        # the tiny CT configuration (64 x 64, 90 angles x 91 bins): a call bound by launches and
        # latency, as parameter studies and tests make it
        _ct("ct64_run", 64, 64, 90, 91, 8),
        # the smallest CT size of the serving mix, block-iterative
        _ct("ct128_bip", 128, 128, 90, 183, 3, mode="bip", blocks=10),
        # the headline: CT 512 x 512, 360 angles x 725 bins, TV, in the one-pass form that the
        # tuner picks for it
        _ct("ct512_run", 512, 512, 360, 725, 6, strategy="one_pass"),
        # the same matrix in a context created with all defaults (bitwise reproducible two-pass
        # sweep), feasibility seeking without perturbation
        _ct("ct512_sweeps", 512, 512, 360, 725, 4, obj="none", call="sweep"),
        # the headline matrix block-iteratively over 36 interleaved angle blocks
        _ct("ct512_bip36", 512, 512, 360, 725, 2, mode="bip", strategy="one_pass", blocks=36),
        # 16-bit matrix storage, the profiling size of the benchmark
        _ct("ct384_f16", 384, 384, 270, 545, 6, dtype="f16", strategy="one_pass"),
        # sparse-view CT of a large image: the perturbation phase weighs as much as the sweep
        _ct("ct1024_sparse", 1024, 1024, 40, 1449, 6, strategy="one_pass"),
        # the extrapolated CT method on an odd-sized image, defaults
        _ct("ct_odd_emr", 301, 217, 181, 397, 4, mode="emr"),
        # sixteen noise realisations of one travel-time survey sharing the matrix; one iteration a
        # call, since the anisotropic subgradient's signs make later ones depend on the last bit
        _seismic("seismic_16rhs", 256, 512, 128, 512, 1, nrhs=16, obj="atv"),
        # one survey on an odd grid with the DROP method
        _seismic("seismic_drop", 199, 333, 97, 301, 6, mode="drop", strategy="one_pass"),
        # the radiotherapy plan, block-iterative over its three structures
        _rt("rt_bip3", 100, 60, 50, 29, 23, 10),
        # the horseshoe plan as a split problem: dose-volume sets by the CQ step, slabs by EMR
        _rt("rt_split", 100, 60, 50, 29, 23, 6, mode="emr", split=True),
    ]


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["ct", "ct", "ct", "seismic", "seismic", "rt"])
    if family == "ct":
        H, W = between(40, 512), between(40, 512)
        if rng.random() < 0.5:
            W = H
        angles, bins = rng.randint(30, 360), max(31, int(1.42 * max(H, W) * rng.uniform(0.7, 1.0)))
        mode = rng.choice(["cimmino", "cimmino", "bip", "drop", "el", "emr"])
        strategy = "default" if mode in ("el", "emr") else rng.choice(["default", "one_pass"])
        blocks = rng.choice([3, 10, 36]) if mode == "bip" else 1
        call = rng.choice(["run", "run", "sweep"])
        c = _ct("", H, W, angles, bins, rng.randint(1, 4), mode=mode, obj="none" if call == "sweep" else "tv",
                dtype=rng.choice(["f32", "f32", "f16", "bf16"]), strategy=strategy,
                blocks=min(blocks, angles), call=call)
    elif family == "seismic":
        H, W = between(48, 256), between(48, 512)
        nrhs = rng.choice([1, 1, 3, 8, 16])
        mode, obj = rng.choice(["cimmino", "drop"]), rng.choice(["tv", "atv"])
        c = _seismic("", H, W, rng.randint(24, 128), rng.randint(60, 512), rng.randint(2, 4) if obj == "tv" else 1,
                     nrhs=nrhs, mode=mode, strategy=rng.choice(["default", "one_pass"]), obj=obj)
    else:
        nx, ny, nz = rng.randint(40, 100), rng.randint(30, 60), rng.randint(20, 50)
        split = rng.random() < 0.5
        c = _rt("", nx, ny, nz, rng.randint(9, 29), rng.randint(8, 23), rng.randint(2, 8),
                mode="emr" if split else "bip", split=split)
    del c["name"]
    return c


# ---------------------------------------------------------------- matrices --

def _trace(px, py, dx, dy, t0, t1, nx, ny, ox, oy, h):
    """CSR of the intersection lengths (float32) of rays p + t d, t in [t0, t1], |d| = 1, with the
    cells of an ny x nx grid of squares: the crossing parameters of the grid lines merged in
    increasing order, each consecutive pair bounding one cell (Siddon's method)."""
    dev = px.device
    kx = ox + h * torch.arange(nx + 1, device=dev, dtype=torch.float64)
    ky = oy + h * torch.arange(ny + 1, device=dev, dtype=torch.float64)
    lens, cols, vals = [], [], []
    chunk = max(1, (1 << 24) // (nx + ny + 2))
    for a in range(0, len(px), chunk):
        s = slice(a, a + chunk)
        p, q, u, v = px[s, None], py[s, None], dx[s, None], dy[s, None]
        lo, hi = t0[s, None], t1[s, None]
        out = torch.zeros_like(lo, dtype=torch.bool)
        spans = []
        for k, c, e in ((kx, p, u), (ky, q, v)):
            flat = e.abs() < 1e-12
            t = (k[None, :] - c) / torch.where(flat, torch.ones_like(e), e)
            first, last = torch.minimum(t[:, :1], t[:, -1:]), torch.maximum(t[:, :1], t[:, -1:])
            lo = torch.where(flat, lo, torch.maximum(lo, first))
            hi = torch.where(flat, hi, torch.minimum(hi, last))
            out |= flat & ((c <= k[0]) | (c >= k[-1]))
            spans.append(torch.where(flat, torch.full_like(t, -1e30), t))
        t = torch.cat([lo, *spans, hi], dim=1)
        t = torch.minimum(torch.maximum(t, lo), hi).sort(dim=1).values
        step = t[:, 1:] - t[:, :-1]
        mid = 0.5 * (t[:, 1:] + t[:, :-1])
        ix = ((p + mid * u - ox) / h).floor().clamp_(0, nx - 1).long()
        iy = ((q + mid * v - oy) / h).floor().clamp_(0, ny - 1).long()
        keep = (step > 1e-9 * h) & (hi > lo) & ~out
        cell = torch.where(keep, iy * nx + ix, torch.full_like(ix, nx * ny))
        cell, order = cell.sort(dim=1)
        step = step.gather(1, order)
        keep = cell < nx * ny
        lens.append(keep.sum(dim=1))
        cols.append(cell[keep].int())
        vals.append(step[keep].float())
    rp = torch.zeros(len(px) + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cat(lens).cumsum(0)
    return rp.int(), torch.cat(cols), torch.cat(vals)


def _rows(csr, idx):
    """The CSR of the rows `idx` of a CSR."""
    rp, col, val = csr
    rp = rp.long()
    ln = rp[idx + 1] - rp[idx]
    out = torch.zeros(len(idx) + 1, dtype=torch.int64, device=rp.device)
    out[1:] = ln.cumsum(0)
    at = torch.arange(int(out[-1]), device=rp.device) + (rp[idx] - out[:-1]).repeat_interleave(ln)
    return out.int(), col[at], val[at]


def _ct_matrix(H, W, angles, bins):
    h = 2.0 / max(H, W)
    r = torch.arange(angles * bins, device="cuda")
    th = (math.pi / angles) * (r // bins).double()
    s = ((r % bins).double() - 0.5 * (bins - 1)) * (h * math.hypot(H, W) / bins)
    big = torch.full_like(s, 1e30)
    return _trace(-s * th.sin(), s * th.cos(), th.cos(), th.sin(), -big, big, W, H,
                  -0.5 * W * h, -0.5 * H * h, h)


def _seismic_matrix(H, W, sources, receivers):
    h = 0.01
    Wk, Hk = W * h, H * h
    sx = (torch.arange(sources, device="cuda", dtype=torch.float64) + 0.5) * Wk / sources
    s = (torch.arange(receivers, device="cuda", dtype=torch.float64) + 0.5) * (2 * Hk + Wk) / receivers
    rx = (s - Hk).clamp(0.0, Wk)
    ry = torch.where(s < Hk, s, torch.where(s < Hk + Wk, torch.full_like(s, Hk), 2 * Hk + Wk - s))
    px = sx.repeat_interleave(receivers)
    ex, ey = rx.repeat(sources) - px, ry.repeat(sources)
    L = torch.hypot(ex, ey)
    return _trace(px, torch.zeros_like(px), ex / L, ey / L, torch.zeros_like(L), L, W, H, 0.0, 0.0, h)


def _rt_plan(nx, ny, nz, beams, ns, nzb):
    """Pencil-beam dose rows of every voxel and the voxels of a horseshoe target, the core organ it
    wraps and a posterior organ; a unit intensity gives a mean target dose of 60."""
    vs, sigma, mu = 3.0, 1.85 * 3.0, 0.004
    cut = 2.35 * sigma
    ds, dz = 0.9 * ny * vs / ns, 0.8 * nz * vs / nzb
    vox = torch.arange(nx * ny * nz, device="cuda")
    X = (vox % nx).double() + 0.5 - nx / 2
    Y = ((vox // nx) % ny).double() + 0.5 - ny / 2
    Z = (vox // (nx * ny)).double() + 0.5 - nz / 2
    px, py, pz = X * vs, Y * vs, Z * vs
    hx, hy = 0.5 * nx * vs, 0.5 * ny * vs
    kp, kq = int(cut / ds) + 1, int(cut / dz) + 1
    cols, vals = [], []
    for b in range(beams):
        th = 2 * math.pi * b / beams
        ux, uy = math.cos(th), math.sin(th)
        depth = torch.full_like(px, math.inf)
        for c, half, e in ((px, hx, ux), (py, hy, uy)):
            if abs(e) > 1e-12:
                depth = torch.minimum(depth, (c + (half if e > 0 else -half)) / e)
        s = py * ux - px * uy
        p0 = (s / ds + 0.5 * (ns - 1)).round().long()
        q0 = (pz / dz + 0.5 * (nzb - 1)).round().long()
        for dq in range(-kq, kq + 1):
            for dp in range(-kp, kp + 1):
                p, q = p0 + dp, q0 + dq
                r2 = (s - (p - 0.5 * (ns - 1)) * ds) ** 2 + (pz - (q - 0.5 * (nzb - 1)) * dz) ** 2
                ok = (r2 < cut * cut) & (p >= 0) & (p < ns) & (q >= 0) & (q < nzb)
                cols.append(torch.where(ok, b * ns * nzb + q * ns + p, torch.full_like(p, -1)).int())
                vals.append((torch.exp(-mu * depth) * torch.exp(-r2 / (2 * sigma * sigma))).float())
    col, val = torch.stack(cols, dim=1), torch.stack(vals, dim=1)
    keep = col >= 0
    rp = torch.zeros(len(vox) + 1, dtype=torch.int64, device="cuda")
    rp[1:] = keep.sum(dim=1).cumsum(0)
    body = (rp.int(), col[keep], val[keep])
    R, zin = torch.hypot(X, Y), Z.abs() < 0.4 * nz
    core = (R < 0.26 * ny) & zin
    shoe = (R >= 0.29 * ny) & (R < 0.39 * ny) & zin & ~((torch.atan2(Y, X) - math.pi / 2).abs() < 0.6)
    post = (Y < -0.36 * ny) & (X.abs() < 0.38 * nx) & ~shoe & ~core
    n = beams * ns * nzb
    parts = [torch.nonzero(k)[:, 0] for k in (shoe, core, post)]
    scale = 60.0 * len(parts[0]) / float(_rows(body, parts[0])[2].double().sum())
    body = (body[0], body[1], body[2] * scale)
    c = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, body[1], body[2].double())
    return body, parts, (c / len(vox)).float(), n


@functools.lru_cache(maxsize=2)
def _geometry(key):
    """The matrix of a case (kept by a user's program for every image or plan taken with it)."""
    c = dict(key)
    if c["family"] == "ct":
        A = _ct_matrix(c["H"], c["W"], c["angles"], c["bins"])
        blocks = (np.arange(c["angles"] * c["bins"]) // c["bins"] % c["blocks"]).astype(np.int32)
        return dict(A=A, n=c["H"] * c["W"], blocks=blocks)
    if c["family"] == "seismic":
        return dict(A=_seismic_matrix(c["H"], c["W"], c["sources"], c["receivers"]), n=c["H"] * c["W"],
                    blocks=None)
    body, (t, o1, o2), lin, n = _rt_plan(c["nx"], c["ny"], c["nz"], c["beams"], c["ns"], c["nzb"])
    kept = (t, o2) if c["split"] else (t, o1, o2)
    blocks = np.repeat(np.arange(len(kept)), [len(k) for k in kept]).astype(np.int32)
    return dict(A=_rows(body, torch.cat(kept)), n=n, blocks=blocks, sizes=[len(k) for k in kept], c=lin,
                Aq=_rows(body, torch.cat((t, o1))), sptr=np.array([0, len(t), len(t) + len(o1)], np.int32))


def _geometry_of(case):
    keys = {"ct": ("family", "H", "W", "angles", "bins", "blocks"),
            "seismic": ("family", "H", "W", "sources", "receivers"),
            "rt": ("family", "nx", "ny", "nz", "beams", "ns", "nzb", "split")}[case["family"]]
    return _geometry(tuple((k, case[k]) for k in keys))


# ------------------------------------------------------------------ inputs --

def _forward(A, x):
    """A x for the float64 image x."""
    rp, col, val = A
    r = torch.zeros(len(rp) - 1, dtype=torch.float64, device=val.device)
    rows = torch.arange(len(r), device=val.device).repeat_interleave((rp[1:] - rp[:-1]).long())
    return r.index_add_(0, rows, val.double() * x[col])


def _phantom(H, W, rng):
    """Ten random ellipses on the grid, clipped to [0, 1]."""
    Y, X = np.meshgrid(-1 + (np.arange(H) + 0.5) * 2 / H, -1 + (np.arange(W) + 0.5) * 2 / W, indexing="ij")
    img = np.zeros((H, W))
    for _ in range(10):
        r, phi = 0.8 * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
        a, b = rng.uniform(0.05, 0.5, size=2)
        th, v = rng.uniform(0, math.pi), rng.uniform(-0.3, 0.6)
        u, w = X - r * math.cos(phi), Y - r * math.sin(phi)
        img[((u * math.cos(th) + w * math.sin(th)) / a) ** 2 + ((w * math.cos(th) - u * math.sin(th)) / b) ** 2 <= 1] += v
    return np.clip(img, 0, 1)


def _slowness(H, W, rng):
    """Slowness (s/km) of wavy layers whose velocity rises with depth from 1.5 to 6 km/s."""
    z, x = (np.arange(H) + 0.5)[:, None] / H, (np.arange(W) + 0.5)[None, :] / W
    layer = np.zeros((H, W), np.int64)
    for k in range(5):
        layer += z > rng.uniform(0.1, 0.9) + 0.05 * np.sin(2 * math.pi * (rng.uniform(0.5, 3) * x + rng.uniform()))
    return 1.0 / np.sort(rng.uniform(1.5, 6.0, 6))[layer]


def _inputs(case, seed):
    """Bounds, box, starting point and constraints of one measurement or plan."""
    geo = _geometry_of(case)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rand = dict(generator=gen, device="cuda", dtype=torch.float64)
    m, n, B = len(geo["A"][0]) - 1, geo["n"], case["nrhs"]
    d = {}
    if case["family"] == "rt":
        sizes = geo["sizes"]
        l = torch.full((m,), -math.inf, device="cuda")
        u = torch.empty(m, device="cuda")
        nt = sizes[0]
        l[:nt], u[:nt] = (57.9, 68.1) if case["split"] else (57.0, 64.2)
        at = nt
        for k, size in enumerate(sizes[1:]):   # the organs' caps differ from plan to plan
            lo = 25.0 if case["split"] or k else 15.0
            u[at:at + size] = rng.uniform(lo, lo + 10)
            at += size
        x0 = 0.5 + torch.rand(n, **rand)
        lo, hi = 0.0, math.inf
        # target D95 >= 60 and D5 <= 65.1, core D5 under its cap
        d["dvcs"] = [(pk.SUPPY_DVC_LOWER, 0, 0.95, 60.0), (pk.SUPPY_DVC_UPPER, 0, 0.05, 65.1),
                     (pk.SUPPY_DVC_UPPER, 1, 0.05, float(rng.uniform(9.0, 12.0)))]
    else:
        ct = case["family"] == "ct"
        img = _phantom(case["H"], case["W"], rng) if ct else _slowness(case["H"], case["W"], rng)
        img = torch.from_numpy(img).cuda().reshape(-1)
        clean = _forward(geo["A"], img)
        if ct:      # low-dose counts
            counts = torch.poisson(5e3 * torch.exp(-clean), generator=gen).clamp_(min=1)
            b = torch.where(clean > 0, -torch.log(counts / 5e3), torch.zeros_like(clean))
            empty = geo["A"][0][1:] == geo["A"][0][:-1]
            b = torch.where(empty, torch.zeros_like(b), b)
            delta, lo, hi = 0.02, 0.0, 1.0
        else:       # travel times with 1% noise, one realisation per right-hand side
            b = clean[:, None] * (1 + 0.01 * torch.randn(m, B, **rand))
            b = b if B > 1 else b[:, 0].contiguous()
            delta, lo, hi = 0.015, 1 / 6.0, 1 / 1.5
        l = torch.minimum(b * (1 - delta), b * (1 + delta)).float()
        u = torch.maximum(b * (1 - delta), b * (1 + delta)).float()
        shape = (n,) if B == 1 else (n, B)
        noise = torch.randn(shape, **rand)
        x0 = (img if B == 1 else img[:, None]) * (1 + 0.1 * noise) + (0.02 if ct else 0.01) * noise.abs()
        x0 = x0.clamp(lo, hi)
    one = lambda v: torch.full((1,), v, device="cuda")  # noqa: E731
    return dict(d, geo=geo, l=l, u=u, x0=x0.float().contiguous(), lo=one(lo), hi=one(hi), m=m, n=n)


def _params(case):
    rt = case["family"] == "rt"
    sup = dict(gamma=1.0, alpha=0.7 if case["split"] else 0.99) if rt else dict(gamma=0.5, alpha=0.99)
    return dict(sup, n_red=1)


def prepare(case, seed):
    d = _inputs(case, seed)
    geo = d["geo"]
    kw = {}
    if case["family"] != "rt":
        kw["shape"] = (case["H"], case["W"])
    if case["obj"] == "mean":
        kw["c_lin"] = geo["c"]
    if case["mode"] == "bip":
        kw["block_of_row"] = geo["blocks"]
    ctx = pk.Context(*geo["A"], d["m"], d["n"], d["l"], d["u"], d["lo"], d["hi"],
                     dtype=DTYPES[case["dtype"]], mode=MODES[case["mode"]], obj=OBJECTIVES[case["obj"]],
                     nrhs=case["nrhs"], strategy=STRATEGIES[case["strategy"]], **kw)
    if case.get("split"):
        ctx.suppy_set_dvc(*geo["Aq"], len(geo["Aq"][0]) - 1, geo["sptr"], d["dvcs"])
    return dict(ctx=ctx, x0=d["x0"], x=torch.empty_like(d["x0"]), call=case["call"], iters=case["iters"],
                params=pk.suppy_params_default(max_sweeps=case["iters"], **_params(case)))


def run(state):
    ctx = state["ctx"]
    ctx.suppy_set_x(state["x0"])
    if state["call"] == "sweep":
        ctx.suppy_sweep(state["params"], state["iters"])
    else:
        ctx.suppy_run(state["params"], want_stats=False)
    ctx.suppy_get_x(state["x"])
    return state["x"]


def work(case):
    """Per iteration the matrix once (values and int32 columns; twice for EMR, whose step length
    needs a second product; the dose matrix of a split problem twice), the bounds and weight of
    every row, the iterate read and written; the perturbation phase reads and writes the iterate
    once more.  Four operations per entry."""
    geo = _geometry_of(case)
    B, m, n = case["nrhs"], len(geo["A"][0]) - 1, geo["n"]
    nnz, vb = len(geo["A"][2]), 4 if case["dtype"] == "f32" else 2
    reads = 2 if case["mode"] == "emr" else 1
    one = reads * nnz * (vb + 4) + m * (8 + 8 * B) + n * 8 * B + (n * 8 * B if case["obj"] != "none" else 0)
    flops = (4 if case["mode"] != "emr" else 6) * nnz * B
    if case.get("split"):
        one += 2 * len(geo["Aq"][2]) * 8
        flops += 4 * len(geo["Aq"][2])
    return {"bytes": case["iters"] * one, "flops": case["iters"] * flops}


# ------------------------------------------------------------ the 64-bit run --

class _Matrix:
    """Products with a CSR matrix in float64, its values rounded to the stored type."""

    def __init__(self, csr, n, dtype="f32"):
        rp, col, val = csr
        val = val.to({"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[dtype])
        self.m, self.n, self.col, self.val = len(rp) - 1, n, col, val.double()
        self.rows = torch.arange(self.m, device=val.device, dtype=torch.int32).repeat_interleave(rp[1:] - rp[:-1])
        self.rho = self._add(self.m, self.rows, self.val * self.val)

    def _add(self, size, at, v):
        return torch.zeros(size, dtype=torch.float64, device=v.device).index_add_(0, at, v)

    def mul(self, x):
        return self._add(self.m, self.rows, self.val * x[self.col])

    def mul_t(self, c):
        return self._add(self.n, self.col, self.val * c[self.rows])


def _objective(case, c):
    """f and a subgradient of the case's objective in float64."""
    if case["obj"] == "mean":
        c = c.double()
        return lambda x: float(c @ x), lambda x: c
    H, W = case["H"], case["W"]

    def tv(x):
        X = x.view(H, W)
        dx, dy = X[1:, :-1] - X[:-1, :-1], X[:-1, 1:] - X[:-1, :-1]
        return dx, dy, torch.sqrt(dx * dx + dy * dy)

    def tv_g(x):
        dx, dy, phi = tv(x)
        inv = torch.where(phi > 0, 1 / phi, torch.zeros_like(phi))
        G = torch.zeros(H, W, dtype=torch.float64, device=x.device)
        G[:-1, :-1] -= (dx + dy) * inv
        G[1:, :-1] += dx * inv
        G[:-1, 1:] += dy * inv
        return G.view(-1)

    def atv(x):
        X = x.view(H, W)
        return float((X[1:] - X[:-1]).abs().sum() + (X[:, 1:] - X[:, :-1]).abs().sum())

    def atv_g(x):
        X = x.view(H, W)
        v, h = torch.sign(X[1:] - X[:-1]), torch.sign(X[:, 1:] - X[:, :-1])
        G = torch.zeros(H, W, dtype=torch.float64, device=x.device)
        G[1:] += v
        G[:-1] -= v
        G[:, 1:] += h
        G[:, :-1] -= h
        return G.view(-1)

    return (lambda x: float(tv(x)[2].sum()), tv_g) if case["obj"] == "tv" else (atv, atv_g)


def _dose_volume(d, dvcs, sptr):
    """sum_j w_j (P_Qj(d) - d): each constraint keeps (upper) or raises (lower) the K highest doses."""
    out = torch.zeros_like(d)
    for kind, s, volume, ref in dvcs:
        a, b = int(sptr[s]), int(sptr[s + 1])
        v = d[a:b]
        K = math.floor(volume * len(v)) if kind == pk.SUPPY_DVC_UPPER else math.ceil(volume * len(v))
        top = torch.zeros_like(v, dtype=torch.bool)
        top[torch.sort(v, descending=True, stable=True).indices[:K]] = True
        move = (~top & (v > ref)) if kind == pk.SUPPY_DVC_UPPER else (top & (v < ref))
        out[a:b] += torch.where(move, ref - v, torch.zeros_like(v)) / len(dvcs)
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    geo, par = d["geo"], _params(case)
    A = _Matrix(geo["A"], d["n"], case["dtype"])
    kept = A.rho > 0
    inv = torch.where(kept, 1 / A.rho, torch.zeros_like(A.rho))
    mode, lo, hi = case["mode"], float(d["lo"]), float(d["hi"])
    block = None
    w = kept.double() / kept.sum()
    if mode == "bip":
        block = torch.from_numpy(geo["blocks"]).long().cuda()
        size = torch.zeros(int(block.max()) + 1, dtype=torch.float64, device="cuda").index_add_(0, block, kept.double())
        w = kept.double() / size[block]
        parts = [torch.nonzero(block == t)[:, 0] for t in range(len(size))]
        parts = [(k, _Matrix(_rows(geo["A"], k), d["n"], case["dtype"])) for k in parts]
    if mode == "drop":
        s = torch.zeros(d["n"], dtype=torch.float64, device="cuda").index_add_(0, A.col, torch.ones_like(A.val))
        z = torch.where(s > 0, 1 / s, torch.zeros_like(s))
    if case["obj"] != "none":
        f, g = _objective(case, geo.get("c"))
    if case.get("split"):
        Q = _Matrix(geo["Aq"], d["n"])
        norms = [float(Q.rho[int(geo["sptr"][s]):int(geo["sptr"][s + 1])].sum()) for _, s, _, _ in d["dvcs"]]
        step = len(norms) / sum(norms)
    done = []
    for k in range(case["nrhs"]):
        pick = (lambda v: v) if case["nrhs"] == 1 else (lambda v: v[:, k])
        l, u, x = pick(d["l"]).double(), pick(d["u"]).double(), pick(d["x0"]).double()
        l, u, x = l.contiguous(), u.contiguous(), x.contiguous()
        ell = 0
        for _ in range(case["iters"]):
            if case["obj"] != "none":
                v = g(x)
                norm, fx = float(v.norm()), f(x)
                for _ in range(100 if norm > 0 else 0):
                    y = x - (par["gamma"] * par["alpha"] ** ell / norm) * v
                    ell += 1
                    if f(y) <= fx:
                        x = y
                        break
            if case.get("split"):
                x = x + step * Q.mul_t(_dose_volume(Q.mul(x), d["dvcs"], geo["sptr"]))
            if mode == "bip":
                for rows, At in parts:
                    r = At.mul(x)
                    x = (x + At.mul_t(w[rows] * inv[rows] * (torch.minimum(torch.maximum(r, l[rows]), u[rows]) - r))).clamp(lo, hi)
                continue
            r = A.mul(x)
            r = torch.minimum(torch.maximum(r, l), u) - r
            if mode == "cimmino":
                x = x + A.mul_t(w * inv * r)
            elif mode == "drop":
                x = x + z * A.mul_t(inv * r)
            else:
                c = w * r * (inv if mode == "el" else 1.0)
                e = A.mul_t(c)
                q = float((w * A.mul(e) ** 2).sum()) if mode == "emr" else float(e @ e)
                t = (float(e @ e) if mode == "emr" else float(r @ c)) / q if q > 0 else 0.0
                x = x + t * e
            x = x.clamp(lo, hi)
        done.append(x)
    return done[0] if case["nrhs"] == 1 else torch.stack(done, dim=1)
