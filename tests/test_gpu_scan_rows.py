"""The raster-row scan (rows of one y each) against the general scan of the same positions, on an S-matrix of
random values, at the edges of its tiles: windows of every size and shape, rows of 3 probes and of more
than one CTA's, steps below a pixel and wider than a window, rows that wrap, run backwards or shift, and
beam sets of one m up to several chunks of pairs."""
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1702_01904_gb300 import prism as P  # noqa: E402
from paper_1702_01904_gb300.runtime import Batch, PrismSimulation  # noqa: E402

pytestmark = pytest.mark.gpu


def plan(n, cell, f, f_y, alpha, seed, precision=P.PRISM_PRECISION_FP32):
    sim = PrismSimulation(P.make_grid(n, n, 1, cell, cell, 2.0, 300.0, f, 2, 0.5, alpha, f_y=f_y, precision=precision))
    i = sim.info
    g = torch.Generator(device="cuda").manual_seed(seed)
    S = torch.randn((i.n_beams, i.ny_s, i.nx_s, 2), generator=g, device="cuda")
    sim.load_smatrix(torch.view_as_complex(S))
    return sim


def close(got, ref, beams, product=0.0):
    # both sum the same products in FP32 in another order: at most one rounding of 2^-24 per beam and per
    # butterfly stage (two transforms of up to 7 stages, and the combinations), twice that for intensities
    # (product: a relative error of every product besides, which add up like the random values do)
    tol = 2.0 * (beams + 24) * 2.0 ** -24 + 2.0 * product * beams ** 0.5
    err = np.linalg.norm(got.astype(np.float64) - ref) / np.linalg.norm(ref)
    assert err <= tol, (err, tol)


def raster(kind, cell, px, py, step):
    x = np.arange(px) * step
    y = np.arange(py) * step * 0.9
    X, Y = np.meshgrid(x, y)
    if kind == "wrap":       # across both cell edges, from negative positions
        X, Y = X - 3.3 * step, Y + cell - 1.7 * step
    elif kind == "serpentine":
        X[1::2] = X[1::2, ::-1]
    elif kind == "skew":     # every row shifted, rows in falling order
        X = X + np.arange(py)[:, None] * 0.37 + 2.0 * cell
        Y = Y[::-1] - 5.0 * cell
    return np.ascontiguousarray(X).ravel(), np.ascontiguousarray(Y).ravel()


@pytest.mark.parametrize("n,cell,f,f_y,alpha", [
    (64, 8.0, 2, 0, 20.0),      # 16 x 16
    (64, 8.0, 2, 1, 20.0),      # 16 x 32
    (128, 12.8, 1, 4, 20.0),    # 64 x 16
    (256, 16.0, 4, 0, 20.0),    # 32 x 32
    (256, 16.0, 4, 2, 9.0),     # 32 x 64
    (256, 12.5, 2, 0, 28.0),    # 64 x 64, 9 pairs of m: two chunks
    (256, 16.0, 1, 0, 14.0),    # 128 x 128
    (256, 16.0, 4, 0, 1.0),     # one beam
])
@pytest.mark.parametrize("kind,px,py,step", [("plain", 3, 9, 0.3), ("wrap", 33, 3, 0.21), ("serpentine", 9, 6, 0.05),
                                             ("skew", 17, 9, 0.4), ("wrap", 7, 4, 2.7), ("plain", 64, 2, 0.11)])
def test_rows_equal_the_general_scan(n, cell, f, f_y, alpha, kind, px, py, step):
    sim = plan(n, cell, f, f_y, alpha, 5)
    x0, y0 = raster(kind, cell, px, py, step)
    probe = P.make_probe(20.0, 30.0, 1.0e6, 1.0e-3, -2.0e-3)
    det = P.make_detector(0.0, 2.0, 40)
    beams = sim.info.n_beams
    got = sim.scan(probe, x0, y0, det, px=px, py=py).cpu().numpy()
    ref = sim.scan(probe, x0, y0, det).cpu().numpy()  # one list of positions: y varies within it
    close(got, ref, beams)
    cb = sim.scan_cbed(probe, x0, y0, px=px, py=py).cpu().numpy()
    close(cb, sim.scan_cbed(probe, x0, y0).cpu().numpy(), beams)
    acc = torch.from_numpy(ref).cuda()
    sim.scan_accumulate(probe, x0, y0, det, 0.5, acc, px=px, py=py)
    close(acc.cpu().numpy(), 1.5 * ref, beams)
    sim.close()


@pytest.mark.parametrize("det", [(0.0, 400.0, 1), (3.0, 0.25, 400), (0.0, 1.0, 4096), (1.0e4, 1.0, 3)])
def test_rows_bins(det):
    # one bin over the whole window, more bins than pixels, lists longer than the windows, empty bins
    sim = plan(256, 16.0, 4, 0, 20.0, 6)
    x0, y0 = raster("wrap", 16.0, 11, 6, 0.3)
    d = P.make_detector(*det)
    got = sim.scan(P.make_probe(20.0), x0, y0, d, px=11, py=6).cpu().numpy()
    ref = sim.scan(P.make_probe(20.0), x0, y0, d).cpu().numpy()
    if ref.any():
        close(got, ref, sim.info.n_beams)
    else:
        assert not got.any()
    sim.close()


def test_rows_partition_and_repeat_bitwise():
    # a probe's result does not depend on the rows scanned with it (bands of rows, single rows), and a
    # second scan on the same plan repeats it; a smaller scan in between changes nothing
    sim = plan(256, 16.0, 4, 0, 20.0, 7)
    x0, y0 = raster("plain", 16.0, 40, 23, 0.3)
    probe, det = P.make_probe(20.0, 12.0), P.make_detector(0.0, 1.0, 100)
    whole = sim.scan(probe, x0, y0, det, px=40, py=23).cpu().numpy()
    sim.scan(probe, x0[:6], y0[:6], det, px=6, py=1)
    assert np.array_equal(sim.scan(probe, x0, y0, det, px=40, py=23).cpu().numpy(), whole)
    for rows in (1, 5):
        for r in range(0, 23, rows):
            k = min(rows, 23 - r)
            part = sim.scan(probe, x0[r * 40:(r + k) * 40], y0[r * 40:(r + k) * 40], det, px=40, py=k).cpu().numpy()
            assert np.array_equal(part, whole[r * 40:(r + k) * 40])
    sim.close()


@pytest.mark.parametrize("n,cell,f,alpha", [(64, 8.0, 2, 20.0), (256, 16.0, 4, 20.0), (256, 12.5, 2, 28.0)])
@pytest.mark.parametrize("kind,px,py,step", [("wrap", 33, 9, 0.21), ("serpentine", 9, 30, 0.05), ("skew", 40, 17, 0.4),
                                             ("plain", 4, 4, 0.3)])
def test_rows_of_value_and_remainder_storage(n, cell, f, alpha, kind, px, py, step):
    # the unpacked S-matrix against the tensor-core scan of the position list, whose products carry 22-bit
    # coefficients and leave out remainder x remainder (2^-22 each, with the 22-bit values at most 2^-20 in all)
    sim = plan(n, cell, f, 0, alpha, 8, P.PRISM_PRECISION_FP16X2)
    x0, y0 = raster(kind, cell, px, py, step)
    probe, det = P.make_probe(20.0, 30.0), P.make_detector(0.0, 2.0, 40)
    got = sim.scan(probe, x0, y0, det, px=px, py=py).cpu().numpy()
    ref = sim.scan(probe, x0, y0, det).cpu().numpy()
    close(got, ref, sim.info.n_beams, 2.0 ** -20)
    cb = sim.scan_cbed(probe, x0, y0, px=px, py=py).cpu().numpy()
    close(cb, sim.scan_cbed(probe, x0, y0).cpu().numpy(), sim.info.n_beams, 2.0 ** -20)
    sim.close()


@pytest.mark.parametrize("precision", [P.PRISM_PRECISION_FP32, P.PRISM_PRECISION_FP16X2])
def test_batch_budget_bounds_the_rows_scratch(precision):
    # a batch over its budget with the rows' scratch fits itself into that of the block scans (fewer rows at
    # once, or blocks), with the results of the batch without a budget to rounding
    n, cell = 256, 12.5
    grid = P.make_grid(n, n, 1, cell, cell, 2.0, 300.0, 2, 2, 0.5, 28.0, precision=precision)
    beams = PrismSimulation(grid).info.n_beams
    V = 50.0 * torch.rand((1, n, n), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")
    x0, y0 = raster("plain", cell, 4, 41, 0.2)
    c = dict(grid=grid, V=V, probe=P.make_probe(20.0), x0=x0, y0=y0, px=4, py=41, det=P.make_detector(0.0, 2.0, 40))
    free = Batch([c])
    free.run()
    free.sync()
    with pytest.raises(P.PrismError) as e:
        Batch([c], hbm_budget_bytes=1)
    least = int(re.search(r"batch needs (\d+) bytes", str(e.value)).group(1))
    assert least < free.info.device_bytes
    with pytest.raises(P.PrismError):
        Batch([c], hbm_budget_bytes=least - 1)
    tight = Batch([c], hbm_budget_bytes=least)
    assert tight.info.device_bytes == least
    tight.run()
    tight.sync()
    close(tight.outs[0].cpu().numpy(), free.outs[0].cpu().numpy().astype(np.float64), beams, 2.0 ** -20)
    free.close()
    tight.close()


@pytest.mark.parametrize("n,cell,f,f_y,alpha", [(64, 8.0, 2, 0, 20.0), (64, 8.0, 2, 1, 20.0), (128, 12.8, 1, 4, 20.0), (256, 16.0, 4, 0, 20.0),
                                                (256, 16.0, 4, 2, 9.0), (256, 12.5, 2, 0, 28.0), (256, 16.0, 1, 0, 14.0), (256, 16.0, 4, 0, 1.0)])
@pytest.mark.parametrize("count", [1, 2, 19, 60, 170])
def test_position_lists(n, cell, f, f_y, alpha, count):
    # probe by probe (one CTA or a cluster of up to 8 per probe) against FP64 sums of the same S-matrix, beams
    # from one to several hundred; positions wrap and are negative
    sim = plan(n, cell, f, f_y, alpha, 9)
    i = sim.info
    r = np.random.default_rng(4)
    x0, y0 = r.uniform(-cell, 2 * cell, count), r.uniform(-cell, 2 * cell, count)
    got = sim.scan_cbed(P.make_probe(20.0, 25.0), x0, y0).cpu().numpy()
    m, k = sim.beams()
    fy = f_y or f
    lam = P.prism_wavelength(300.0)
    qx, qy = m * f / cell, k * fy / cell
    inside = (lam * qx) ** 2 + (lam * qy) ** 2 <= 0.02 ** 2 * (1 + 1e-12)
    A = inside * np.exp(-1j * np.pi * lam * (qx ** 2 + qy ** 2) * 25.0)
    S = sim.smatrix().cpu().numpy().astype(np.complex128)
    for p in sorted({0, count // 2, count - 1}):
        a = A * np.exp(-2j * np.pi * (qx * x0[p] + qy * y0[p]))
        ix = (int(np.floor(x0[p] / (cell / i.nx_s) + 0.5)) - i.nw_x // 2 + np.arange(i.nw_x)) % i.nx_s
        iy = (int(np.floor(y0[p] / (cell / i.ny_s) + 0.5)) - i.nw_y // 2 + np.arange(i.nw_y)) % i.ny_s
        psi = np.tensordot(a, S[:, iy[:, None], ix[None, :]], axes=(0, 0))
        ref = np.abs(np.fft.fft2(psi)) ** 2 / ((i.nw_x * i.nw_y) ** 2 * inside.sum())
        # (the FP32 coefficients besides: phase and product, 2^-22 of each)
        close(got[p], ref, i.n_beams, 2.0 ** -22)
    det = P.make_detector(0.0, 2.0, 40)
    out = sim.scan(P.make_probe(20.0, 25.0), x0, y0, det).cpu().numpy()
    wx = np.fft.fftfreq(i.nw_x, 1.0 / i.nw_x) * f / cell
    wy = np.fft.fftfreq(i.nw_y, 1.0 / i.nw_y) * fy / cell
    b = np.floor(1000.0 * lam * np.sqrt(wx[None, :] ** 2 + wy[:, None] ** 2) / 2.0).astype(int)
    ref = np.stack([got[:, b == j].astype(np.float64).sum(1) for j in range(40)], axis=1)
    close(out, ref, i.n_beams)
    sim.close()
