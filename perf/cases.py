"""What this library is measured on: calls a STEM simulation program makes, over the sizes it makes them at.

A program builds the S-matrix of a cell (prism_build_smatrix, from device or pinned host potentials),
scans probe rasters against the resident S-matrix many times (annular detectors or full diffraction
patterns, FP32 or 16-bit storage), or runs conventional multislice per probe.  The cells are those of
the repository's workloads (256^2 simple-cubic cell, 512^2 nanoparticle cell, 1024^2 amorphous carbon,
2048^2 serving cell): 300 kV, 20 mrad, 2 Angstrom slices, random-atom potentials of their density.
"""
import math

import numpy as np
import torch

from paper_1702_01904_gb300 import prism as P
from paper_1702_01904_gb300.runtime import PrismSimulation, multislice

KV, DZ, ALPHA = 300.0, 2.0, 20.0
PRECISIONS = {"fp32": P.PRISM_PRECISION_FP32, "fp16": P.PRISM_PRECISION_FP16, "bf16": P.PRISM_PRECISION_BF16,
              "fp16x2": P.PRISM_PRECISION_FP16X2}


def _case(call, n, cell, slices, f=4, f_y=0, px=0, py=0, step=0.25, raster=True, precision="fp32", bins=100, step_mrad=1.0,
          c1=0.0, c3=0.0, tilt=0.0):
    return dict(call=call, n=n, cell=cell, slices=slices, f=f, f_y=f_y, px=px, py=py, step=step, raster=raster,
                precision=precision, bins=bins, step_mrad=step_mrad, c1=c1, c3=c3, tilt=tilt)


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # one region of a small resident cell: an interactive scan or a small serving request
        named("scan-256", "scan", 256, 16.0, 8, 4, px=16, py=16, step=1.0),
        # S-matrix of a small cell: one of many in a parameter study (launches and latency)
        named("build-256", "build", 256, 16.0, 8, 4),
        # conventional multislice of a small cell, the reference a PRISM result is checked against
        named("multislice-256", "multislice", 256, 16.0, 8, px=16, py=16, step=1.0),
        # 4D-STEM of a jittered (not raster) ptychography scan with separate factors f_x, f_y
        named("cbed-512-rect", "cbed", 512, 32.0, 18, 8, f_y=16, px=900, py=1, raster=False, c1=60.0),
        # a ragged region with compact FP32-class storage, aberrated and tilted probe
        named("scan-512-fp16x2", "scan", 512, 32.0, 18, 4, px=33, py=31, precision="fp16x2", c1=50.0, c3=1.0e7, tilt=2.0),
        # a whole simulation through host buffers: potential in, detector stack out (213 beams)
        named("host-512", "host", 512, 32.0, 18, 4, px=32, py=32),
        # the full raster of the 1024^2 amorphous-carbon cell from its resident S-matrix
        named("scan-1024", "scan", 1024, 50.0, 50, 8, px=200, py=200),
        # the same raster from a 16-bit S-matrix
        named("scan-1024-fp16", "scan", 1024, 50.0, 50, 8, px=200, py=200, precision="fp16"),
        # S-matrix of that cell: 129 beams through 50 slices
        named("build-1024", "build", 1024, 50.0, 50, 8),
        # region-of-interest scan of the large serving cell (529 beams, 128-pixel windows)
        named("scan-2048", "scan", 2048, 102.4, 6, 8, px=32, py=32, step=0.35),
        # S-matrix of the large serving cell, a thin section of it
        named("build-2048", "build", 2048, 102.4, 6, 8),
        # conventional multislice of the amorphous-carbon cell
        named("multislice-1024", "multislice", 1024, 50.0, 50, px=10, py=10, step=2.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        call = rng.choice(["scan", "scan", "scan", "cbed", "build", "build", "host", "multislice"])
        n = rng.choice([128, 256, 512, 1024, 2048])
        cell = round(n * rng.choice([0.0488, 0.05, 0.0625]), 3)
        f = rng.choice([f for f in (2, 4, 8, 16) if 16 <= n // 2 // f <= 128 and n // 2 // f * f * 2 == n])
        nw = n // 2 // f
        precision, f_y = "fp32", 0
        if call in ("scan", "cbed"):
            if nw <= 64:
                precision = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16", "fp16x2"])
            if precision == "fp32" and nw in (16, 32) and rng.random() < 0.15:
                f_y = f // 2  # windows of nw x 2 nw pixels
        beams = len(_beams(n, cell, f, f_y)[0])
        if precision == "fp16x2" and beams > 370:
            precision = "fp32"
        slices = _log_int(rng, 2, 60) if call in ("build", "host", "multislice") else rng.randint(1, 6)
        raster = call == "multislice" or rng.random() < 0.85
        px, py = _log_int(rng, 1, 220), _log_int(rng, 1, 220)
        if not raster:
            px, py = px * py, 1
        step = round(math.exp(rng.uniform(math.log(0.1), math.log(1.0))), 3)
        bins, step_mrad = rng.choice([(100, 1.0), (100, 1.0), (40, 2.5), (3, 30.0), (1, 400.0)])
        c = _case(call, n, cell, slices, f, f_y, px, py, step, raster, precision, bins, step_mrad,
                  c1=rng.choice([0.0, 0.0, round(rng.uniform(-100, 100), 1)]), c3=rng.choice([0.0, 0.0, 1.0e7]),
                  tilt=rng.choice([0.0, 0.0, 0.0, round(rng.uniform(0.5, 5.0), 2)]))
        probes = px * py
        # no more work than the largest listed cases: propagated pixels, direct beam-sum products, outputs
        waves = 0 if call in ("scan", "cbed") else probes if call == "multislice" else beams
        prods = 0 if call in ("build", "multislice") else probes * beams * nw * (nw if not f_y else 2 * nw)
        if waves * slices * n * n > 7e9 or (call != "multislice" and beams * slices * n * n > 9e9):
            continue
        if prods > 2.2e10 or (call == "cbed" and probes * nw * nw > 6e7):
            continue
        return c


# ---------------------------------------------------------------- inputs
def _potential(case, seed):
    """Projected potentials [slices][n][n] float32 (V Angstrom) on the GPU: 0.1 atoms per cubic Angstrom
    at random pixels, each a Gaussian of 0.3 Angstrom width and 25 Z^0.7 peak (Z = 6, and 29 for a tenth)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, h, cell = case["n"], case["slices"], case["cell"]
    atoms = max(1, int(round(0.1 * cell * cell * DZ)))
    k = torch.fft.fftfreq(n, d=cell / n, device="cuda", dtype=torch.float64)
    k = torch.where(k > 0.5 * n / cell, k - n / cell, k)
    kx = torch.fft.rfftfreq(n, d=cell / n, device="cuda", dtype=torch.float64)
    sg = 0.3
    blur = (torch.exp(-2.0 * (math.pi * sg) ** 2 * (k[:, None] ** 2 + kx[None, :] ** 2)) * (2.0 * math.pi * sg * sg) * (n / cell) ** 2)
    blur = blur.to(torch.float32)
    out = torch.empty((h, n, n), dtype=torch.float32, device="cuda")
    for p in range(h):
        where = torch.randint(0, n * n, (atoms,), generator=g, device="cuda")
        heavy = torch.rand(atoms, generator=g, device="cuda") < 0.1
        grid = torch.bincount(where[~heavy], minlength=n * n).to(torch.float32) * (25.0 * 6.0 ** 0.7)
        grid += torch.bincount(where[heavy], minlength=n * n).to(torch.float32) * (25.0 * 29.0 ** 0.7)
        out[p] = torch.fft.irfft2(torch.fft.rfft2(grid.reshape(n, n)) * blur, s=(n, n)).clamp_(min=0.0)
    return out


def _positions(case, seed):
    """Probe positions in Angstrom: a raster from a random corner, or scattered over the cell."""
    r = np.random.default_rng([seed, 17])
    px, py, cell = case["px"], case["py"], case["cell"]
    if not case["raster"]:
        return r.uniform(0.0, cell, px * py), r.uniform(0.0, cell, px * py)
    ox, oy = r.uniform(0.0, cell, 2)
    x, y = np.meshgrid(ox + case["step"] * np.arange(px), oy + case["step"] * np.arange(py))
    return x.ravel(), y.ravel()


class _DeviceView:
    """The plan's S-matrix in place; holds on to the simulation whose memory it is."""

    def __init__(self, sim):
        i = sim.info
        self.sim = sim
        self.__cuda_array_interface__ = {"data": (P.prism_plan_smatrix(sim.plan), False), "typestr": "<f4", "version": 3,
                                         "shape": (i.n_beams, i.ny_s, i.nx_s, 2)}


def prepare(case, seed):
    s = {"case": case}
    n, cell, call = case["n"], case["cell"], case["call"]
    grid = P.make_grid(n, n, case["slices"], cell, cell, DZ, KV, case["f"], 2, 0.5, ALPHA, precision=PRECISIONS[case["precision"]],
                       f_y=case["f_y"])
    V = _potential(case, seed)
    torch.cuda.synchronize()
    s["grid"] = grid
    s["probe"] = P.make_probe(ALPHA, case["c1"], case["c3"], 1e-3 * case["tilt"], 0.0)
    s["det"] = P.make_detector(0.0, case["step_mrad"], case["bins"])
    if case["px"]:
        s["x0"], s["y0"] = _positions(case, seed)
    if call == "multislice":
        s["V"] = V
        return s
    sim = s["sim"] = PrismSimulation(grid)
    if call == "build":
        s["V"] = V
    elif call == "host":
        s["V"] = V.cpu().pin_memory()
        s["out"] = torch.empty((case["px"] * case["py"], case["bins"]), dtype=torch.float32).pin_memory()
    else:
        sim.build(V)
        sim.sync()
        sim._V = None
    if call in ("build", "host"):
        s["S"] = torch.as_tensor(_DeviceView(sim), device="cuda")
    return s


def run(s):
    c = s["case"]
    call = c["call"]
    if call == "multislice":
        return multislice(s["grid"], s["V"], s["probe"], s["x0"], s["y0"], s["det"], px=c["px"], py=c["py"])
    sim = s["sim"]
    if call == "build":
        sim.build(s["V"])
        return s["S"]
    if call == "host":
        sim.build_host(s["V"])
        sim.scan_host(s["probe"], s["x0"], s["y0"], s["det"], s["out"], px=c["px"], py=c["py"])
        return s["S"], s["out"]
    if call == "cbed":
        return sim.scan_cbed(s["probe"], s["x0"], s["y0"], px=c["px"], py=c["py"])
    return sim.scan(s["probe"], s["x0"], s["y0"], s["det"], px=c["px"], py=c["py"])


# ---------------------------------------------------------------- work
def _wavelength():
    h, m, e, c = 6.62607015e-34, 9.1093837015e-31, 1.602176634e-19, 299792458.0
    ev = e * KV * 1e3
    return h / math.sqrt(2.0 * m * ev * (1.0 + ev / (2.0 * m * c * c))) * 1e10


def _sigma():
    h, m, e, c = 6.62607015e-34, 9.1093837015e-31, 1.602176634e-19, 299792458.0
    return 2.0 * math.pi * (m + e * KV * 1e3 / (c * c)) * e * (_wavelength() * 1e-10) / (h * h) * 1e-10


def _beams(n, cell, f, f_y):
    """(m, n) of the plane waves (m f, n f_y) / cell inside the aperture, n-major."""
    fy = f_y or f
    lam, a = _wavelength(), ALPHA * 1e-3
    mm, nm = int(a / (lam * f / cell)) + 1, int(a / (lam * fy / cell)) + 1
    y, x = np.meshgrid(np.arange(-nm, nm + 1), np.arange(-mm, mm + 1), indexing="ij")
    inside = (lam * (x * f) / cell) ** 2 + (lam * (y * fy) / cell) ** 2 <= a * a * (1.0 + 1e-12)
    return x[inside], y[inside]


def work(case):
    n, h, px, py, f = case["n"], case["slices"], case["px"], case["py"], case["f"]
    f_y = case["f_y"] or f
    m, _ = _beams(n, case["cell"], f, case["f_y"])
    beams, probes, nw, nwy = len(m), px * py, n // 2 // f, n // 2 // f_y
    pot, smat = 4.0 * h * n * n, 8.0 * beams * (n // 2) ** 2
    # a slice: two row transforms of n rows, two column transforms of the n / 2 columns inside the
    # anti-aliasing aperture, the transmission and the propagator products
    slice_flops = 10.0 * n * n * math.log2(n) * 1.5 + 9.0 * n * n
    # a window: the beam sum (on a raster row the beams of one m share their y phase, so each probe
    # sums its distinct m; scattered probes sum every beam) and the window transform
    terms = len(set(m.tolist())) if case["raster"] else beams
    window = nw * nwy * (8.0 * terms + 5.0 * math.log2(nw * nwy) + 3.0)
    out = probes * 4.0 * (nw * nwy if case["call"] == "cbed" else case["bins"])
    # S-matrix pixels under the windows
    reach = 2.0 * case["cell"] / n
    rx, ry = ((nw + (px - 1) * case["step"] / reach, nwy + (py - 1) * case["step"] / reach) if case["raster"] else (n / 2, n / 2))
    seen = min(n / 2, rx) * min(n / 2, ry) / (n / 2) ** 2
    store = {"fp32": 1.0, "fp16x2": 1.0, "fp16": 0.5, "bf16": 0.5}[case["precision"]]
    if case["call"] == "build":
        return {"bytes": pot + smat, "flops": beams * h * slice_flops}
    if case["call"] == "host":
        return {"bytes": pot + smat + out, "flops": beams * h * slice_flops + probes * window}
    if case["call"] == "multislice":
        return {"bytes": pot + out, "flops": probes * h * slice_flops}
    return {"bytes": smat * seen * store + 16.0 * probes + out, "flops": probes * window}


# ---------------------------------------------------------------- in 64 bits
def _freq(n):
    return np.concatenate([np.arange(n // 2), np.arange(-(n // 2), 0)]).astype(np.float64)


def _dev(a, dtype=torch.complex128):
    return torch.as_tensor(a, device="cuda").to(dtype)


def _propagator(case):
    n, cell = case["n"], case["cell"]
    q = _freq(n) / cell
    q2 = q[:, None] ** 2 + q[None, :] ** 2
    q_aa = 0.5 * (0.5 * n / cell)
    return _dev(np.exp(-1j * math.pi * _wavelength() * DZ * q2) * (q2 < q_aa * q_aa))


def _aperture(case, qx, qy):
    """Aperture and aberrations of the (tilted) probe at (qx, qy), and its shift at the exit surface."""
    lam = _wavelength()
    t = 1e-3 * case["tilt"]
    dx = qx - t / lam
    inside = (lam * dx) ** 2 + (lam * qy) ** 2 <= (ALPHA * 1e-3) ** 2 * (1.0 + 1e-12)
    q2 = dx * dx + qy * qy
    chi = math.pi * lam * q2 * case["c1"] + 0.5 * math.pi * lam ** 3 * q2 * q2 * case["c3"]
    return inside * np.exp(-1j * chi), DZ * case["slices"] * math.tan(t)


def _propagate(psi, V, prop, sigma):
    for p in range(V.shape[0]):
        psi = torch.fft.ifft2(torch.fft.fft2(psi * torch.exp(1j * sigma * V[p].double())) * prop)
    return psi


def _smatrix(case, V):
    n, f, fy = case["n"], case["f"], case["f_y"] or case["f"]
    m, k = _beams(n, case["cell"], f, case["f_y"])
    prop, sigma = _propagator(case), _sigma()
    S = torch.empty((len(m), n // 2, n // 2), dtype=torch.complex128, device="cuda")
    r = np.arange(n)
    step = max(1, int(3e8 // (16 * n * n)))
    for b in range(0, len(m), step):
        ex = _dev(np.exp(2j * math.pi * ((m[b:b + step, None] * f * r) % n) / n))
        ey = _dev(np.exp(2j * math.pi * ((k[b:b + step, None] * fy * r) % n) / n))
        psi = _propagate(ey[:, :, None] * ex[:, None, :], V, prop, sigma)
        S[b:b + step] = psi[:, ::2, ::2]  # band-limited to |k| < n / 4: every second sample
    return S, m, k


def _bins(case, qx, qy):
    theta = 1000.0 * _wavelength() * np.sqrt(qx * qx + qy * qy)
    b = np.floor(theta / case["step_mrad"]).astype(np.int64)
    return torch.as_tensor(np.where(b < case["bins"], b, case["bins"]).ravel(), device="cuda")


def _summed(case, inten, bins):
    out = torch.zeros((inten.shape[0], case["bins"] + 1), dtype=torch.float64, device="cuda")
    out.index_add_(1, bins, inten.reshape(inten.shape[0], -1))
    return out[:, :case["bins"]]


def _scan(case, S, m, k, x0, y0):
    n, cell, f, fy = case["n"], case["cell"], case["f"], case["f_y"] or case["f"]
    nd, nwx, nwy = n // 2, n // 2 // f, n // 2 // fy
    qx, qy = m * f / cell, k * fy / cell
    A, shift = _aperture(case, qx, qy)
    norm = float(np.sum(np.abs(A) ** 2))
    sx = (np.floor(x0 / (cell / nd) + 0.5).astype(np.int64) - nwx // 2) % nd
    sy = (np.floor(y0 / (cell / nd) + 0.5).astype(np.int64) - nwy // 2) % nd
    wx, wy = _freq(nwx) * f / cell, _freq(nwy) * fy / cell
    bins = _bins(case, wx[None, :], wy[:, None])
    flat = S.reshape(len(m), -1)
    outs = []
    step = max(1, int(6e8 // (16 * len(m) * nwx * nwy)))
    for p in range(0, len(x0), step):
        e = slice(p, p + step)
        a = _dev(A[None, :] * np.exp(-2j * math.pi * (qx[None, :] * (x0[e, None] - shift) + qy[None, :] * y0[e, None])))
        iy = torch.as_tensor((sy[e, None] + np.arange(nwy)) % nd, device="cuda")
        ix = torch.as_tensor((sx[e, None] + np.arange(nwx)) % nd, device="cuda")
        win = flat[:, (iy[:, :, None] * nd + ix[:, None, :]).reshape(len(a), -1)]  # [beams][probes][pixels]
        psi = torch.einsum("pb,bpw->pw", a, win).reshape(len(a), nwy, nwx)
        inten = torch.fft.fft2(psi).abs() ** 2 / ((nwx * nwy) ** 2 * norm)
        outs.append(inten if case["call"] == "cbed" else _summed(case, inten, bins))
    return torch.cat(outs)


def _multislice(case, V, x0, y0):
    n, cell = case["n"], case["cell"]
    q = _freq(n) / cell
    qx, qy = np.broadcast_to(q[None, :], (n, n)), np.broadcast_to(q[:, None], (n, n))
    A, shift = _aperture(case, qx, qy)
    norm = float(np.sum(np.abs(A) ** 2))
    bins, prop, sigma, A = _bins(case, qx, qy), _propagator(case), _sigma(), _dev(A)
    outs = []
    step = max(1, int(3e8 // (16 * n * n)))
    for p in range(0, len(x0), step):
        e = slice(p, p + step)
        ex = _dev(np.exp(-2j * math.pi * q[None, :] * (x0[e, None] - shift)))
        ey = _dev(np.exp(-2j * math.pi * q[None, :] * y0[e, None]))
        psi = _propagate(torch.fft.ifft2(A[None] * ey[:, :, None] * ex[:, None, :]), V, prop, sigma)
        outs.append(_summed(case, torch.fft.fft2(psi).abs() ** 2 / norm, bins))
    return torch.cat(outs)


def exact(case, seed):
    V = _potential(case, seed)
    x0, y0 = _positions(case, seed) if case["px"] else (None, None)
    if case["call"] == "multislice":
        return _multislice(case, V, x0, y0)
    S, m, k = _smatrix(case, V)
    if case["call"] == "build":
        return torch.view_as_real(S)
    out = _scan(case, S, m, k, x0, y0)
    return (torch.view_as_real(S), out) if case["call"] == "host" else out
