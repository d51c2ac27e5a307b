"""Performance cases: reconstructions as a program that uses this library runs them.

Every case goes through the public binding (paper_2608_28183_gb300.nlos): plans
are made once per capture shape and autotuned, as the README's example does,
and a pass reconstructs a capture that is on the device into a volume buffer
the program keeps. `exact` restates each path in float64 with plain torch.
"""
from __future__ import annotations

import math

import torch

from paper_2608_28183_gb300 import nlos

C_LIGHT = 299_792_458.0
TAPER_BINS = 8.0
TICKS_PER_BIN, T0_TICKS = 16, 1000


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(kind, nx, ny, nt, storage="f32", **kw):
    return dict(kind=kind, nx=nx, ny=ny, nt=nt, storage=storage, **kw)


def listed():
    return [
        # live preview of a coarse 32 x 32 scan: a few microseconds a stage, launches count
        dict(_case("fk", 32, 32, 256), name="fk_32x32x256_f32"),
        # the same kind of preview with phasor fields, 40 planes
        dict(_case("pf", 32, 32, 512, depths=40), name="pf_32x32x512_f32"),
        # a scan whose grid is no power of two and not square, 300 bins
        dict(_case("fk", 96, 80, 300), name="fk_96x80x300_f32"),
        # mid-size capture, long time axis, half-precision storage as the server runs it
        dict(_case("fk", 128, 128, 1024, "f16"), name="fk_128x128x1024_f16"),
        # the headline f-k workload
        dict(_case("fk", 256, 256, 512), name="fk_256x256x512_f32"),
        # the sizes of the paper's exhaustive captures (190 x 190 points, 3002 bins): the largest call
        dict(_case("fk", 190, 190, 3002), name="fk_190x190x3002_f32"),
        # the phasor-field workload: 128 planes, 151 band frequencies
        dict(_case("pf", 128, 128, 1024, depths=128), name="pf_128x128x1024_f32"),
        # the densest phasor-field capture of the batch mix, half-precision storage
        dict(_case("pf", 256, 256, 512, "f16", depths=128), name="pf_256x256x512_f16"),
        # one frame of a dynamic capture: 1.2 M photon records to phasors to a volume
        dict(_case("photons", 128, 128, 1024, depths=128, photons=1_200_000), name="photons_128x128x1024_1.2M"),
        # mixture of experts: both reconstructions from one spectrum, images, mix
        dict(_case("moe", 128, 128, 1024, depths=128), name="moe_128x128x1024"),
        # temporal merging of four complex volumes, and the display image
        dict(_case("merge", 256, 256, 512, frames=4), name="merge_256x256x512_4"),
        # mixed captures (two sides, both methods, two of each) replayed as one CUDA graph
        dict(_case("batch", 128, 128, 512, "f16", depths=128), name="batch_8_mixed_f16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _storage(rng):
    return rng.choice(["f32", "f32", "f32", "f16", "f16", "bf16"])


def draw(rng):
    kind = rng.choice(["fk", "fk", "fk", "pf", "pf", "photons", "moe", "merge", "batch"])
    pow2 = rng.random() < 0.5          # half the scans are on power-of-two grids, as the workloads are

    def side(lo, hi):
        return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi))) if pow2 else _log_int(rng, lo, hi)

    if kind == "fk":
        nx = side(8, 256)
        ny = nx if rng.random() < 0.6 else side(8, 256)
        nt = 1 << rng.randint(7, 10) if pow2 else _log_int(rng, 100, 1024)
        c = _case("fk", nx, ny, nt, _storage(rng))
        if rng.random() < 0.15:
            c["output"] = "complex"
        elif pow2 and min(nx, ny) >= 16 and rng.random() < 0.2:
            c["pad"] = 1
        return c
    if kind == "merge":
        return _case("merge", side(32, 256), side(32, 256), _log_int(rng, 128, 512), frames=rng.randint(2, 8))
    if kind == "batch":
        s = rng.choice([32, 48, 64, 96, 128])
        return _case("batch", s, s, rng.choice([256, 400, 512]), rng.choice(["f16", "f16", "f32"]),
                     depths=rng.randint(24, 128))
    nx = side(16, 128)
    ny = nx if rng.random() < 0.6 else min(128, max(16, round(nx * rng.uniform(0.5, 1.5))))
    nt = 1 << rng.randint(8, 10) if pow2 else _log_int(rng, 256, 1024)
    depths = rng.choice([40, 64, 128, 128, _log_int(rng, 16, 160)])
    if kind == "pf":
        c = _case("pf", nx, ny, nt, rng.choice(["f32", "f32", "f16"]), depths=depths)
        if rng.random() < 0.15:
            c["output"] = "complex"
        return c
    if kind == "photons":
        return _case("photons", nx, ny, nt, depths=depths, photons=_log_int(rng, 50_000, 5_000_000))
    return _case("moe", nx, ny, nt, depths=depths)


# ---------------------------------------------------------------------------
# geometry shared by prepare, work and exact
# ---------------------------------------------------------------------------

def _geometry(nx, ny, nt):
    """1 m walls at 32 ps for coarse scans, 2 m at 16 ps otherwise; square
    wall cells, so a non-square grid is a non-square wall."""
    w, dt = (1.0, 32e-12) if max(nx, ny) <= 48 else (2.0, 16e-12)
    cell = w / max(nx, ny)
    return nlos.Geometry(nx, ny, nt, dt, cell * nx, cell * ny)


def _depths(g, depths):
    far = g.nt * C_LIGHT * g.bin_width_s / 2.0
    lo = 0.4
    return dict(n_depths=depths, depth_min_m=lo, depth_max_m=max(far, 2 * lo))


def _pow2(x):
    return 1 << max(0, math.ceil(math.log2(x)))


def _dtype(storage):
    return {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[storage]


def _items(case):
    """Captures of a batch: (method, side, nt) of the eight reconstructions, two of each shape."""
    s = case["nx"]
    shapes = [("fk", s), ("pf", s), ("fk", s // 2), ("pf", s // 2)]
    return [(m, n, case["nt"], k) for m, n in shapes for k in range(2)]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _expected(g, gen):
    """Expected photon counts of a hidden scene (points and two tilted plates)
    in front of the wall, plus a background of half a count per bin."""
    dev = "cuda"
    f64 = dict(dtype=torch.float64, device=dev)
    far = 0.9 * g.nt * C_LIGHT * g.bin_width_s / 2.0
    u = torch.rand((10, 4), generator=gen, **f64)
    span = torch.tensor([g.wall_w_m, g.wall_h_m], **f64)
    pts = [torch.cat([(u[:, :2] - 0.5) * 0.8 * span, 0.2 * far + 0.7 * far * u[:, 2:3], 0.3 + 0.7 * u[:, 3:]], 1)]
    grid = torch.linspace(-0.5, 0.5, 5, **f64)
    for _ in range(2):
        v = torch.rand(6, generator=gen, **f64)
        p = torch.zeros((25, 4), **f64)
        p[:, 0] = (v[0] - 0.5) * 0.5 * span[0] + (grid[:, None] * 0.3 * span[0]).expand(5, 5).reshape(-1)
        p[:, 1] = (v[1] - 0.5) * 0.5 * span[1] + (grid[None, :] * 0.3 * span[1]).expand(5, 5).reshape(-1)
        p[:, 2] = (0.3 + 0.5 * v[2]) * far + (v[3] - 0.5) * p[:, 0]
        p[:, 2].clamp_(min=0.15 * far)
        p[:, 3] = 0.05 + 0.1 * v[4]
        pts.append(p)
    x = (torch.arange(g.nx, **f64) + 0.5) * (g.wall_w_m / g.nx) - g.wall_w_m / 2
    y = (torch.arange(g.ny, **f64) + 0.5) * (g.wall_h_m / g.ny) - g.wall_h_m / 2
    vol = torch.zeros(g.nx * g.ny * g.nt, dtype=torch.float32, device=dev)
    row = torch.arange(g.nx * g.ny, device=dev).reshape(g.nx, g.ny) * g.nt
    for px, py, pz, al in torch.cat(pts).tolist():
        r = torch.sqrt((x[:, None] - px) ** 2 + (y[None, :] - py) ** 2 + pz * pz)
        b = torch.floor(2.0 * r / (C_LIGHT * g.bin_width_s)).long()
        w = torch.where(b < g.nt, al / r ** 4, torch.zeros_like(r)).float()
        at = (row + b.clamp(max=g.nt - 1)).reshape(-1)      # one bin per wall point: no two alike
        vol[at] += w.reshape(-1)
    peak = 10.0 ** (2.0 + float(torch.rand(1, generator=gen, **f64)))
    return (vol * (peak / vol.max().clamp(min=1e-30)) + 0.5).reshape(g.nx, g.ny, g.nt)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)


def _transient(g, storage, seed):
    gen = _generator(seed)
    return torch.poisson(_expected(g, gen), generator=gen).to(_dtype(storage))


def _photon_records(g, count, seed):
    """About `count` records in scan order, as a scanning capture delivers them."""
    gen = _generator(seed)
    lam = _expected(g, gen)
    counts = torch.poisson(lam * (count / float(lam.double().sum())), generator=gen).reshape(-1).long()
    idx = torch.repeat_interleave(torch.arange(counts.numel(), device="cuda"), counts)
    jitter = torch.randint(0, TICKS_PER_BIN, (idx.numel(),), generator=gen, device="cuda")
    ticks = T0_TICKS + (idx % g.nt) * TICKS_PER_BIN + jitter
    return (idx // g.nt).int().view(torch.uint32), ticks.int().view(torch.uint32)


def _frames(case, seed):
    gen = _generator(seed)
    shape = (case["nx"], case["ny"], case["nt"])

    def field():
        return torch.view_as_complex(torch.randn(shape + (2,), generator=gen, device="cuda"))
    still = field() * torch.rand(shape, generator=gen, device="cuda") ** 4
    return [still + 0.2 * field() for _ in range(case["frames"])]


# ---------------------------------------------------------------------------
# what a program keeps, and one pass
# ---------------------------------------------------------------------------

def _plan(method, g, case, **kw):
    p = nlos.plan_for_capture(g, method, case["storage"], **kw)
    p.autotune()
    return p


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "merge":
        st["frames"] = _frames(case, seed)
        shape = st["frames"][0].shape
        st["merged"] = torch.empty(shape, device="cuda")
        st["coherence"] = torch.empty(shape, device="cuda")
        st["image"] = torch.empty(shape[:2], device="cuda")
        return st
    if kind == "batch":
        plans, ins, outs = [], [], []
        for j, (m, n, nt, k) in enumerate(_items(case)):
            g = _geometry(n, n, nt)
            if k == 0:
                plan = _plan(m, g, case, **(_depths(g, case["depths"]) if m == "pf" else {}))
            plans.append(plan)
            ins.append(_transient(g, case["storage"], seed * 16 + j))
            outs.append(plan.empty_volume())
        st.update(outs=outs, batch=nlos.Batch(plans, ins, outs))
        return st
    g = _geometry(case["nx"], case["ny"], case["nt"])
    out = dict(output=case["output"]) if "output" in case else {}
    if kind == "fk":
        st["plan"] = _plan("fk", g, case, pad_factor=case.get("pad", 2), **out)
        st["x"] = _transient(g, case["storage"], seed)
        st["vol"] = st["plan"].empty_volume()
        return st
    st["plan"] = _plan("pf", g, case, **_depths(g, case["depths"]), **out)
    st["vol"] = st["plan"].empty_volume()
    if kind == "photons":
        st["pixel"], st["ticks"] = _photon_records(g, case["photons"], seed)
        st["phasors"] = st["plan"].empty_phasors()
        return st
    st["x"] = _transient(g, case["storage"], seed)
    if kind == "moe":
        st["fk"] = _plan("fk", g, case)
        st["vol_fk"] = st["fk"].empty_volume()
        st["stream2"] = torch.cuda.Stream()
        st["images"] = [torch.empty((g.nx, g.ny), device="cuda") for _ in range(3)]
    return st


def run(st):
    kind = st["kind"]
    if kind in ("fk", "pf"):
        return st["plan"].reconstruct(st["x"], st["vol"])
    if kind == "photons":
        ph = st["plan"].bin_phasors(st["pixel"], st["ticks"], T0_TICKS, TICKS_PER_BIN, phasors=st["phasors"])
        return [ph, st["plan"].reconstruct_phasors(ph, st["vol"])]
    if kind == "moe":
        vf, vp = nlos.reconstruct_moe(st["fk"], st["plan"], st["x"], st["vol_fk"], st["vol"], stream2=st["stream2"])
        a = nlos.max_image(vf, take_sqrt=True, image=st["images"][0])
        b = nlos.max_image(vp, image=st["images"][1])
        return [vf, vp, a, b, nlos.moe_mix(a, b, out=st["images"][2])]
    if kind == "merge":
        m, c = nlos.coherence_merge(st["frames"], merged=st["merged"], coherence=st["coherence"])
        return [m, c, nlos.max_image(m, image=st["image"])]
    st["batch"].launch()
    return st["outs"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _fft_flops(count, n):
    return 5.0 * count * n * math.log2(n) if n > 1 else 0.0


def _band(g):
    """(Lt, df, f0, k_lo, F, sigma_f) of the plan's virtual wave (4 cells, 5 cycles)."""
    lt = _pow2(g.nt)
    f0 = C_LIGHT / (4.0 * g.wall_w_m / g.nx)
    df = 1.0 / (lt * g.bin_width_s)
    k0 = math.floor(f0 / df + 0.5)
    sigma_f = 6.0 * f0 / (2.0 * math.pi * 5.0)
    kh = math.floor(5.0 * sigma_f / df + 0.5)
    lo, hi = max(1, k0 - kh), min(lt // 2 - 1, k0 + kh)
    return lt, df, f0, lo, hi - lo + 1, sigma_f


def _radial_counts(g, k_hi_freq):
    dx, dy = g.wall_w_m / g.nx, g.wall_h_m / g.ny
    nu, nv = _pow2(2 * g.nx), _pow2(2 * g.ny)
    r_max = math.hypot(0.5 * nu * dx, 0.5 * nv * dy)
    rho_max = math.hypot(0.5 / dx, 0.5 / dy)
    lam = C_LIGHT / k_hi_freq
    n_r = max(2, _pow2(math.ceil(4.0 * r_max / lam - 1e-9) + 1))
    n_rho = _pow2(math.ceil(2.0 * r_max * rho_max - 1e-9) + 1)
    return nu, nv, r_max, rho_max, n_r, n_rho


def _work_fk(g, storage, out_bytes, pad=2, shared=False):
    a, b, n = g.nx, g.ny, g.nt
    lx, ly, lt = (a, b, n) if pad == 1 else (_pow2(2 * a), _pow2(2 * b), _pow2(2 * n))
    hx, m = lx // 2 + 1, lt // 2
    fl = 0.0 if shared else _fft_flops(b * n, lx) / 2 + _fft_flops(hx * n, ly)
    fl += _fft_flops(hx * ly, lt) + 20.0 * lx * ly * min(n, m)
    fl += _fft_flops(lx * min(n, m), ly) + _fft_flops(b * min(n, m), lx) + _fft_flops(a * b, lt)
    v = a * b * n
    return (0 if shared else v * _dtype(storage).itemsize) + v * out_bytes, fl


def _work_pf(g, storage, depths, out_bytes, source="transient"):
    lt, df, _, lo, F, _ = _band(g)
    nu, nv, _, _, _, n_rho = _radial_counts(g, (lo + F - 1) * df)
    a, b, D = g.nx, g.ny, depths
    eb = 8 if storage == "f32" else 4
    by = n_rho * F * D * eb + a * b * D * out_bytes     # the radial kernel and the volume
    fl = _fft_flops(a * F, nv) + _fft_flops(nv * F, nu) + 8.0 * nu * nv * F * D
    fl += _fft_flops(nu * D, nv) + _fft_flops(b * D, nu)
    if source == "transient":
        by += a * b * g.nt * _dtype(storage).itemsize
        fl += _fft_flops(a * b, lt) / 2
    elif source == "phasors":
        by += a * b * F * 8
    return by, fl


def work(case):
    kind = case["kind"]
    g = _geometry(case["nx"], case["ny"], case["nt"])
    v = g.nx * g.ny * g.nt
    ob = 8 if case.get("output") == "complex" else 4
    if kind == "fk":
        by, fl = _work_fk(g, case["storage"], ob, case.get("pad", 2))
    elif kind == "pf":
        by, fl = _work_pf(g, case["storage"], case["depths"], ob)
    elif kind == "photons":
        by, fl = _work_pf(g, "f32", case["depths"], 4, "phasors")
        F, lt = _band(g)[4], _band(g)[0]
        by += 8 * case["photons"]
        fl += min(4.0 * case["photons"] * F, _fft_flops(g.nx * g.ny, lt) / 2)
    elif kind == "moe":
        by, fl = _work_fk(g, "f32", 4)
        by2, fl2 = _work_pf(g, "f32", case["depths"], 4, "spectrum")
        by, fl = by + by2 + 12 * g.nx * g.ny, fl + fl2
    elif kind == "merge":
        by, fl = v * (8 * case["frames"] + 8) + 4 * g.nx * g.ny, v * (8.0 * case["frames"] + 8)
    else:
        by, fl = 0.0, 0.0
        for m, n, nt, _ in _items(case):
            h = _geometry(n, n, nt)
            x, y = _work_fk(h, case["storage"], 4) if m == "fk" else _work_pf(h, case["storage"], case["depths"], 4)
            by, fl = by + x, fl + y
    return {"bytes": float(by), "flops": float(fl)}


# ---------------------------------------------------------------------------
# the same results in float64, in plain torch
# ---------------------------------------------------------------------------

def _exact_fk(H, g, pad=2, complex_out=False):
    a, b, n = g.nx, g.ny, g.nt
    lx, ly, lt = (a, b, n) if pad == 1 else (_pow2(2 * a), _pow2(2 * b), _pow2(2 * n))
    half = lt // 2
    ar = dict(dtype=torch.float64, device="cuda")
    ramp = torch.arange(n, **ar) / (n - 1)
    U = torch.fft.fft2((H.double() * ramp).to(torch.complex128), s=(lx, ly), dim=(0, 1))     # [lx][ly][n]
    sx = C_LIGHT * g.bin_width_s / (2.0 * g.wall_w_m / a)
    sy = C_LIGHT * g.bin_width_s / (2.0 * g.wall_h_m / b)
    X = torch.fft.fftfreq(lx, 1.0 / lx, **ar) / (lx // 2) * sx
    Y = torch.fft.fftfreq(ly, 1.0 / ly, **ar) / (ly // 2) * sy
    Z = torch.arange(1, half, **ar) / half
    for k in range(lx):
        S = torch.fft.fft(U[k], n=lt, dim=1)[:, :half]
        zp = torch.sqrt(X[k] ** 2 + (Y ** 2)[:, None] + (Z ** 2)[None, :])
        mu = half * zp
        ok = mu <= half - 1
        k0 = torch.where(ok, torch.floor(mu), torch.zeros_like(mu)).long()
        al = torch.where(ok, mu - k0, torch.zeros_like(mu))
        k1 = (k0 + 1).clamp(max=half - 1)
        V = torch.zeros((ly, lt), dtype=torch.complex128, device="cuda")
        V[:, 1:half] = torch.where(ok, ((1 - al) * S.gather(1, k0) + al * S.gather(1, k1)) * (Z / zp), 0)
        U[k] = torch.fft.ifft(V, dim=1)[:, :n]
    psi = torch.fft.ifft(torch.fft.ifft(U, dim=1)[:, :b], dim=0)[:a]
    return psi.contiguous() if complex_out else psi.real ** 2 + psi.imag ** 2


def _exact_phasors(H, g):
    lt, _, _, lo, F, _ = _band(g)
    return torch.fft.rfft(H.double(), n=lt, dim=2)[:, :, lo:lo + F]


def _exact_pf(P, g, depths, weighted=False, complex_out=False):
    """Radial Rayleigh-Sommerfeld operator on phasors P[x][y][F] (w(f) applied here unless `weighted`)."""
    ar = dict(dtype=torch.float64, device="cuda")
    lt, df, f0, lo, F, sigma_f = _band(g)
    freqs = (lo + torch.arange(F, **ar)) * df
    w = torch.exp(-(freqs - f0) ** 2 / (2.0 * sigma_f ** 2))
    kappa = 2.0 * math.pi * freqs / C_LIGHT
    nu, nv, r_max, rho_max, n_r, n_rho = _radial_counts(g, (lo + F - 1) * df)
    dd = _depths(g, depths)
    d = torch.full((1,), dd["depth_min_m"], **ar) if depths == 1 else \
        dd["depth_min_m"] + torch.arange(depths, **ar) * ((dd["depth_max_m"] - dd["depth_min_m"]) / (depths - 1))
    dr = r_max / (n_r - 1)
    r = torch.arange(n_r, **ar) * dr
    q = torch.full((n_r,), dr, **ar)
    q[0] = q[-1] = 0.5 * dr
    rho = torch.arange(n_rho, **ar) * (rho_max / (n_rho - 1))
    rho_cut = min(rho_max, 0.5 * (n_r - 1) / r_max)
    rc = rho_cut * (n_rho - 1) / rho_max
    B = q * 2.0 * math.pi * r * torch.special.bessel_j0(2.0 * math.pi * r[None, :] * rho[:, None])
    B[rho > rho_cut] = 0.0
    ph = 2.0 * kappa[None, :, None] * torch.sqrt(r[:, None, None] ** 2 + d[None, None, :] ** 2)
    A = torch.polar(torch.ones_like(ph), ph).reshape(n_r, -1)
    K = torch.complex(B @ A.real.contiguous(), B @ A.imag.contiguous()).reshape(n_rho, F, depths)
    Ph = torch.fft.fft2(P.to(torch.complex128) if weighted else P * w, s=(nu, nv), dim=(0, 1)).reshape(nu * nv, F)
    fx = torch.fft.fftfreq(nu, g.wall_w_m / g.nx, **ar)
    fy = torch.fft.fftfreq(nv, g.wall_h_m / g.ny, **ar)
    rb = (torch.sqrt(fx[:, None] ** 2 + fy[None, :] ** 2) * ((n_rho - 1) / rho_max)).reshape(-1)
    t = (rc - rb) / TAPER_BINS
    taper = torch.where(rb <= rc - TAPER_BINS, 1.0, torch.where(rb >= rc, 0.0, t * t * (3.0 - 2.0 * t)))
    ic = math.floor(rc)
    i0 = torch.floor(rb).long().clamp(0, max(0, min(ic - 1, n_rho - 2)))
    al = rb - i0
    C = torch.zeros((nu * nv, depths), dtype=torch.complex128, device="cuda")
    order = torch.argsort(i0)
    ends = torch.cumsum(torch.bincount(i0, minlength=n_rho), 0).tolist()
    start = 0
    for i, end in enumerate(ends):
        if end > start:
            px = order[start:end]
            a = al[px, None]
            C[px] = taper[px, None] * ((1 - a) * (Ph[px] @ K[i]) + a * (Ph[px] @ K[min(i + 1, ic)]))
        start = end
    I = torch.fft.ifft2(C.reshape(nu, nv, depths), dim=(0, 1))[:g.nx, :g.ny]
    return I.contiguous() if complex_out else I.abs()


def exact(case, seed):
    kind = case["kind"]
    cpx = case.get("output") == "complex"
    if kind == "merge":
        f = [x.to(torch.complex128) for x in _frames(case, seed)]
        s = sum(f).abs()
        c = s / (1e-6 + sum(x.abs() for x in f))
        m = c * s / len(f)
        return [m, c, m.amax(dim=2)]
    if kind == "batch":
        out = []
        for j, (m, n, nt, _) in enumerate(_items(case)):
            g = _geometry(n, n, nt)
            H = _transient(g, case["storage"], seed * 16 + j)
            out.append(_exact_fk(H, g) if m == "fk" else _exact_pf(_exact_phasors(H, g), g, case["depths"]))
        return out
    g = _geometry(case["nx"], case["ny"], case["nt"])
    if kind == "photons":
        pixel, ticks = (t.view(torch.int32).long() for t in _photon_records(g, case["photons"], seed))
        flat = pixel * g.nt + (ticks - T0_TICKS) // TICKS_PER_BIN
        H = torch.bincount(flat, minlength=g.nx * g.ny * g.nt).reshape(g.nx, g.ny, g.nt)
        _, df, f0, lo, F, sigma_f = _band(g)
        fr = (lo + torch.arange(F, dtype=torch.float64, device="cuda")) * df
        P = _exact_phasors(H, g) * torch.exp(-(fr - f0) ** 2 / (2.0 * sigma_f ** 2))
        return [P, _exact_pf(P, g, case["depths"], weighted=True)]
    H = _transient(g, case["storage"], seed)
    if kind == "fk":
        return _exact_fk(H, g, case.get("pad", 2), cpx)
    vp = _exact_pf(_exact_phasors(H, g), g, case["depths"], complex_out=cpx)
    if kind == "pf":
        return vp
    vf = _exact_fk(H, g)
    a, b = vf.amax(dim=2).sqrt(), vp.amax(dim=2)
    mix = a / a.max() * (b / b.max() + 1e-3) ** 0.3
    return [vf, vp, a, b, mix / mix.max()]
