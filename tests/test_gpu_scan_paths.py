"""Every kernel that a scan can take, with the path asserted: the block scan's contraction shapes, split blocks,
work-unit counters, scratch and shared-memory limits on positions that go by blocks (rasters of many probes
whose rows do not share a y, tall rasters of two columns)."""
import ctypes
import re
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1702_01904_gb300 import prism as P  # noqa: E402
from paper_1702_01904_gb300.runtime import Batch, PrismSimulation  # noqa: E402

pytestmark = pytest.mark.gpu

DET = P.make_detector(0.0, 2.0, 40)
PROBE = P.make_probe(20.0, 12.0)


def plan(n, cell, f, seed, f_y=0, alpha=20.0, precision=P.PRISM_PRECISION_FP32, budget=0):
    sim = PrismSimulation(P.make_grid(n, n, 1, cell, cell, 2.0, 300.0, f, 2, 0.5, alpha, f_y=f_y, precision=precision), budget)
    i = sim.info
    g = torch.Generator(device="cuda").manual_seed(seed)
    sim.load_smatrix(torch.view_as_complex(torch.randn((i.n_beams, i.ny_s, i.nx_s, 2), generator=g, device="cuda")))
    return sim


def jittered(px, py, step, seed=0):
    # a raster whose probes are off their row by up to a quarter of a step, across the cell's edges
    r = np.random.default_rng(seed)
    x, y = np.meshgrid(step * np.arange(px) - 1.3, step * np.arange(py) - 0.7)
    return x.ravel(), (y + 0.25 * step * r.uniform(-1.0, 1.0, y.shape)).ravel()


def scan(sim, pos, px, py, path):
    out = sim.scan(PROBE, *pos, DET, px=px, py=py).cpu().numpy()
    assert P.prism_plan_scan_path(sim.plan) == path
    return out


def exact(sim, cell, f, f_y, x0, y0):
    """Bins of the probes in 64 bits."""
    i = sim.info
    m, k = sim.beams()
    f_y = f_y or f
    lam = P.prism_wavelength(300.0)
    qx, qy = m * f / cell, k * f_y / cell
    inside = (lam * qx) ** 2 + (lam * qy) ** 2 <= 0.02 ** 2 * (1 + 1e-12)
    A = inside * np.exp(-1j * np.pi * lam * (qx ** 2 + qy ** 2) * 12.0)
    S = sim.smatrix().cpu().numpy().astype(np.complex128)
    wx, wy = (np.fft.fftfreq(n, 1.0 / n) * ff / cell for n, ff in ((i.nw_x, f), (i.nw_y, f_y)))
    b = np.floor(1000.0 * lam * np.sqrt(wx[None, :] ** 2 + wy[:, None] ** 2) / 2.0).astype(int)
    out = []
    for x, y in zip(x0, y0):
        a = A * np.exp(-2j * np.pi * (qx * x + qy * y))
        ix = (int(np.floor(x / (cell / i.nx_s) + 0.5)) - i.nw_x // 2 + np.arange(i.nw_x)) % i.nx_s
        iy = (int(np.floor(y / (cell / i.ny_s) + 0.5)) - i.nw_y // 2 + np.arange(i.nw_y)) % i.ny_s
        psi = np.tensordot(a, S[:, iy[:, None], ix[None, :]], axes=(0, 0))
        inten = np.abs(np.fft.fft2(psi)) ** 2 / ((i.nw_x * i.nw_y) ** 2 * inside.sum())
        out.append([inten[b == j].sum() for j in range(40)])
    return np.array(out)


def close(got, ref, beams):
    # one rounding of 2^-24 per beam, butterfly stage and combination at most, an FP32 coefficient of 2^-22
    # per product besides, twice that for intensities
    err = np.linalg.norm(got.astype(np.float64) - ref) / np.linalg.norm(ref)
    assert err <= 2.0 * ((beams + 24) * 2.0 ** -24 + 2.0 ** -22 * beams ** 0.5), err


# windows of 16, 32 and 64 pixels; sides that leave partial blocks of 4 x 8, 8 x 4 and 2 x 16
@pytest.mark.parametrize("n,cell,f,px,py,step", [(128, 8.0, 4, 101, 97, 0.11), (128, 12.8, 2, 53, 49, 0.2), (512, 32.0, 4, 47, 45, 0.1)])
def test_block_scan_in_every_contraction_shape(n, cell, f, px, py, step):
    sim = plan(n, cell, f, 1)
    pos = jittered(px, py, step)
    ref = scan(sim, pos, px, py, P.PRISM_SCAN_BLOCKS)
    some = np.array([0, px - 1, 7 * px + 5, px * py // 2, px * py - 1])
    close(ref[some], exact(sim, cell, f, 0, pos[0][some], pos[1][some]), sim.info.n_beams)
    shapes = P.prism_plan_tune_result(sim.plan, P.PRISM_TUNE_SCAN).n_shapes
    assert shapes == 6
    for v in range(shapes):
        sim.set_shape(P.PRISM_TUNE_SCAN, v)
        assert np.array_equal(scan(sim, pos, px, py, P.PRISM_SCAN_BLOCKS), ref), P.prism_tune_shape_name(P.PRISM_TUNE_SCAN, v)
    sim.set_shape(P.PRISM_TUNE_SCAN, -1)
    out = sim.autotune_scan(PROBE, *pos, DET, px=px, py=py).cpu().numpy()
    assert P.prism_plan_scan_path(sim.plan) == P.PRISM_SCAN_BLOCKS and np.array_equal(out, ref)
    ms = sim.tune_result()["scan"]["ms"]
    assert len(set(ms.values())) > 1 and ms[sim.tune_result()["scan"]["chosen"]] == min(ms.values())
    sim.close()


@pytest.mark.parametrize("f,f_y", [(8, 4), (4, 8), (4, 2)])
def test_block_scan_of_unequal_windows(f, f_y):
    # 16 x 32, 32 x 16 and 32 x 64 pixels
    sim = plan(256, 16.0, f, 2, f_y=f_y)
    px, py = 83, 90
    pos = jittered(px, py, 0.13)
    out = scan(sim, pos, px, py, P.PRISM_SCAN_BLOCKS)
    some = np.array([0, px - 1, px * py - 1])
    close(out[some], exact(sim, 16.0, f, f_y, pos[0][some], pos[1][some]), sim.info.n_beams)
    sim.close()


@pytest.mark.parametrize("shape", range(6))
def test_block_scan_grows_its_scratch_for_each_shape(shape):
    # a small first scan by blocks, then a pinned shape and a larger raster
    n, cell, f = 128, 12.8, 2
    small, pos = jittered(40, 52, 0.2, 3), jittered(101, 99, 0.1, 4)
    sim = plan(n, cell, f, 3)
    ref = scan(sim, pos, 101, 99, P.PRISM_SCAN_BLOCKS)
    sim.close()
    sim = plan(n, cell, f, 3)
    scan(sim, small, 40, 52, P.PRISM_SCAN_BLOCKS)
    sim.set_shape(P.PRISM_TUNE_SCAN, shape)
    assert np.array_equal(scan(sim, pos, 101, 99, P.PRISM_SCAN_BLOCKS), ref)
    sim.close()


def test_block_scan_bands_and_repeats_bitwise():
    # 320 blocks of 4 x 8 (more than the CTAs: the last round is split) against bands of 16 rows (80 blocks,
    # all split), on one plan in turn: the split changes no bit and the work-unit counters, whose place moves
    # with the grid, are left zero
    sim = plan(128, 12.8, 2, 5)
    pos = jittered(160, 64, 0.09, 5)
    whole = scan(sim, pos, 160, 64, P.PRISM_SCAN_BLOCKS)
    for r in range(0, 64, 16):
        e = slice(r * 160, (r + 16) * 160)
        band = scan(sim, (pos[0][e], pos[1][e]), 160, 16, P.PRISM_SCAN_BLOCKS)
        assert np.array_equal(band, whole[e])
        assert np.array_equal(scan(sim, pos, 160, 64, P.PRISM_SCAN_BLOCKS), whole)
    sim.close()


def test_block_scan_of_two_columns():
    x, y = np.meshgrid(0.2 + 0.2 * np.arange(2), 0.05 * np.arange(1040))
    sim = plan(128, 12.8, 2, 6)
    out = scan(sim, (x.ravel(), y.ravel()), 2, 1040, P.PRISM_SCAN_BLOCKS)
    some = np.array([0, 1, 1039, 2079])
    close(out[some], exact(sim, 12.8, 2, 0, x.ravel()[some], y.ravel()[some]), sim.info.n_beams)
    sim.close()


def test_block_scans_of_different_beam_counts_at_once():
    # the shared-memory limit of one kernel, from four threads with plans of different beam counts
    sims = [plan(256, 16.0, 4, 7 + i, alpha=a) for i, a in enumerate((20.0, 15.0, 28.0, 18.0))]
    assert len({s.info.n_beams for s in sims}) == 4
    pos = jittered(65, 63, 0.2, 7)
    refs = [scan(s, pos, 65, 63, P.PRISM_SCAN_BLOCKS) for s in sims]
    outs, errors = [None] * 4, []

    def worker(i):
        try:
            for _ in range(5):
                o = sims[i].scan(PROBE, *pos, DET, px=65, py=63)
                sims[i].sync()
            outs[i] = o.cpu().numpy()
        except Exception as e:  # reported below
            errors.append(e)

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=300)
    assert not errors, errors
    for s, o, r in zip(sims, outs, refs):
        assert np.array_equal(o, r)
        s.close()


def test_list_bins_are_added_in_64_bits():
    # the bins of scattered probes with 64-pixel windows against FP64 sums of their diffraction patterns: one beam
    # in the aperture, so that the normalisation 2^-24 is exact.  A bin of at most 32 pixels is four FP32 sums
    # of three additions' depth, added in FP64 and rounded: (1 + 1/2 + 1/4) / 4 + 1 roundings' variance, 1.2 rms,
    # and the patterns' own add little; five additions deep in FP32 and then rounded it would be 1.71.  Half way
    # between: 1.45, a rounding of 2^-24 being 0.425 rms (uniform, mantissas spread over their logarithm).
    sim = plan(512, 32.0, 4, 8)
    i = sim.info
    r = np.random.default_rng(8)
    pos = (r.uniform(0.0, 32.0, 400), r.uniform(0.0, 32.0, 400))
    probe = P.make_probe(1.0)
    inten = sim.scan_cbed(probe, *pos).cpu().numpy().reshape(400, -1).astype(np.float64)
    assert P.prism_plan_scan_path(sim.plan) == P.PRISM_SCAN_LIST
    out = sim.scan(probe, *pos, P.make_detector(0.0, 1.0, 100)).cpu().numpy()
    assert P.prism_plan_scan_path(sim.plan) == P.PRISM_SCAN_LIST
    w = np.fft.fftfreq(i.nw_x, 1.0 / i.nw_x) * 4 / 32.0
    b = np.floor(1000.0 * i.wavelength * np.sqrt(w[None, :] ** 2 + w[:, None] ** 2)).astype(int).ravel()
    err = np.concatenate([out[:, k] / inten[:, b == k].sum(1) - 1.0 for k in range(100) if 12 <= (b == k).sum() <= 32])
    assert err.size > 5000
    assert np.sqrt(np.mean(err ** 2)) <= 1.45 * 0.425 * 2.0 ** -24
    sim.close()


@pytest.mark.parametrize("n,cell,f,f_y", [(128, 8.0, 4, 0), (128, 12.8, 2, 0), (256, 16.0, 8, 4), (256, 16.0, 4, 8)])
def test_list_equals_blocks_bitwise(n, cell, f, f_y):
    # windows of up to 1024 pixels: probes from a raster that goes by blocks, scanned as a list (long enough that
    # no two CTAs share a probe's beams)
    sim = plan(n, cell, f, 9, f_y=f_y)
    pos = jittered(101, 97, 0.11, 9)
    whole = scan(sim, pos, 101, 97, P.PRISM_SCAN_BLOCKS)
    some = np.random.default_rng(9).choice(101 * 97, 300, replace=False)
    part = scan(sim, (pos[0][some], pos[1][some]), 300, 1, P.PRISM_SCAN_LIST)
    assert np.array_equal(part, whole[some])
    sim.close()


def test_list_sums_over_beams():
    # 64-pixel windows, 213 beams of independent random values: no further from 64 bits than the block scan's two
    # sums.  Each of those is rounded once per beam at a size growing as the root of the beams summed: B / 2
    # roundings' variance against the whole, a rounding of 2^-24 being 0.425 rms; 20 more for the coefficients
    # and two transforms of 6 stages.  One chain rounded twice per beam has B of them.
    sim = plan(512, 32.0, 4, 10)
    i = sim.info
    r = np.random.default_rng(10)
    x, y = r.uniform(0.0, 32.0, 300), r.uniform(0.0, 32.0, 300)  # (long enough that no two CTAs share a probe's beams)
    out = sim.scan_cbed(P.make_probe(20.0), x, y).cpu().numpy()
    assert P.prism_plan_scan_path(sim.plan) == P.PRISM_SCAN_LIST
    m, k = sim.beams()
    qx, qy = m * 4 / 32.0, k * 4 / 32.0
    S = sim.smatrix().cpu().numpy().astype(np.complex128)
    num = den = 0.0
    for p in range(0, 300, 10):
        a = np.exp(-2j * np.pi * (qx * x[p] + qy * y[p]))
        ix = (int(np.floor(x[p] / 0.125 + 0.5)) - 32 + np.arange(64)) % 256
        iy = (int(np.floor(y[p] / 0.125 + 0.5)) - 32 + np.arange(64)) % 256
        ref = np.abs(np.fft.fft2(np.tensordot(a, S[:, iy[:, None], ix[None, :]], axes=(0, 0)))) ** 2 / (4096.0 ** 2 * len(m))
        num += np.sum((out[p] - ref) ** 2)
        den += np.sum(ref ** 2)
    assert i.n_beams == len(m) == 213
    assert np.sqrt(num / den) <= 0.425 * 2.0 ** -24 * np.sqrt(213 / 2 + 20)
    sim.close()


@pytest.mark.parametrize("n,cell,f,px,py,step,path", [
    (512, 32.0, 4, 16, 16, 0.1, P.PRISM_SCAN_LIST),      # 213 beams, 64-pixel windows: few probes
    (512, 32.0, 4, 40, 40, 0.1, P.PRISM_SCAN_BLOCKS),    # blocks that share tiles
    (512, 32.0, 4, 4, 200, 0.25, P.PRISM_SCAN_BLOCKS),
    (512, 32.0, 4, 40, 40, 11.0, P.PRISM_SCAN_LIST),     # windows further apart than that
    (128, 12.8, 2, 45, 45, 0.1, P.PRISM_SCAN_BLOCKS),    # 137 beams, 32-pixel windows
    (256, 16.0, 4, 30, 30, 0.3, P.PRISM_SCAN_LIST),      # 49 beams
    (128, 8.0, 4, 101, 97, 0.1, P.PRISM_SCAN_BLOCKS),    # 13 beams, 16-pixel windows
    (1024, 50.0, 4, 10, 1, 0.3, P.PRISM_SCAN_LIST),      # 505 beams, 128-pixel windows
    (1024, 50.0, 4, 20, 1, 0.3, P.PRISM_SCAN_BLOCKS),
])
def test_jittered_rasters_take_the_faster_path(n, cell, f, px, py, step, path):
    sim = plan(n, cell, f, 11)
    pos = jittered(px, py, step, 11)
    out = scan(sim, pos, px, py, path)
    some = np.array([0, px * py // 2, px * py - 1])
    close(out[some], exact(sim, cell, f, 0, pos[0][some], pos[1][some]), sim.info.n_beams)
    sim.close()


@pytest.mark.parametrize("n,cell,f,px,py,step", [
    (512, 32.0, 8, 4, 99, 0.6),     # 32-pixel windows: the blocks' scratch holds one row at a time
    (512, 32.0, 4, 3, 75, 0.31),    # 64-pixel windows, 213 beams
    (128, 12.8, 2, 6, 6, 0.1),      # partial blocks, all split
])
@pytest.mark.parametrize("budget,path", [(0, P.PRISM_SCAN_ROWS), (1 << 33, P.PRISM_SCAN_TENSOR)])
def test_narrow_value_and_remainder_rasters(n, cell, f, px, py, step, budget, path):
    # by rows in one or two launches where memory is free, else by tensor-core blocks in split mode: never in many
    # launches of a few rows
    # a raster by tensor-core blocks in split mode or by rows, against 64 bits: 22-bit values and coefficients, and
    # remainder x remainder left out, are at most 2^-20 of each product
    sim = plan(n, cell, f, 12, precision=P.PRISM_PRECISION_FP16X2, budget=budget)
    x, y = np.meshgrid(step * np.arange(px) - 1.3, step * np.arange(py) - 0.7)
    pos = (x.ravel(), y.ravel())
    out = scan(sim, pos, px, py, path)
    some = np.array([0, px - 1, px * py // 2, px * py - 1])
    ref = exact(sim, cell, f, 0, pos[0][some], pos[1][some])
    err = np.linalg.norm(out[some] - ref) / np.linalg.norm(ref)
    assert err <= 2.0 * (2.0 ** -20 * sim.info.n_beams ** 0.5 + (sim.info.n_beams + 24) * 2.0 ** -24), err
    before = sim.launches()
    assert np.array_equal(scan(sim, pos, px, py, path), out)
    assert sim.launches() - before <= (5 if path == P.PRISM_SCAN_ROWS else 1)
    sim.close()


@pytest.mark.parametrize("py", [1, 2, 3])
def test_few_rows_of_small_value_and_remainder_windows(py):
    sim = plan(128, 8.0, 4, 13, precision=P.PRISM_PRECISION_FP16X2)
    x, y = np.meshgrid(0.2 * np.arange(47), 0.2 * np.arange(py))
    pos = (x.ravel(), y.ravel())
    out = scan(sim, pos, 47, py, P.PRISM_SCAN_TENSOR if py <= 2 else P.PRISM_SCAN_ROWS)
    ref = exact(sim, 8.0, 4, 0, *pos)
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) <= 2.0 * (2.0 ** -20 * 13 ** 0.5 + (13 + 24) * 2.0 ** -24)
    sim.close()


@pytest.mark.parametrize("px,py", [(11, 9), (7, 16), (1, 130), (130, 1)])
def test_positions_are_checked_everywhere(px, py):
    # a NaN, an infinity or a position beyond 2^28 pixels anywhere among them is refused; the largest position
    # allowed, and rows whose y are zeros of both signs, are not
    sim = plan(128, 8.0, 4, 14)
    x, y = np.meshgrid(0.2 * np.arange(px), 0.2 * np.arange(py))
    pos = [x.ravel(), y.ravel()]
    ref = sim.scan(PROBE, *pos, DET, px=px, py=py).cpu().numpy()
    path = P.prism_plan_scan_path(sim.plan)
    for axis in (0, 1):
        for at in sorted({0, 1, 5, px * py // 2, px * py - 2, px * py - 1}):
            for bad in (np.nan, -np.nan, np.inf, -np.inf, 2.0 ** 28 * 0.125 * (1 + 2.0 ** -50), -1e300):
                p = [q.copy() for q in pos]
                p[axis][at] = bad
                with pytest.raises(P.PrismError) as e:
                    sim.scan(PROBE, *p, DET, px=px, py=py)
                assert e.value.status == P.PRISM_ERR_INVALID
    p = [q.copy() for q in pos]
    p[1][: px : 2] = -0.0
    assert np.array_equal(sim.scan(PROBE, *p, DET, px=px, py=py).cpu().numpy(), ref)
    assert P.prism_plan_scan_path(sim.plan) == path
    p[0][:] = 2.0 ** 28 * 0.125
    sim.scan(PROBE, *p, DET, px=px, py=py)
    sim.close()


@pytest.mark.parametrize("precision", [P.PRISM_PRECISION_FP32, P.PRISM_PRECISION_FP16X2])
def test_a_plan_holds_the_scratch_of_one_path(precision):
    # a plan that scans by rows and by blocks in turn keeps one scratch, as large as the larger needs
    def held(sim):
        return P.prism_plan_info(sim.plan).device_bytes

    x, y = np.meshgrid(0.2 * np.arange(60), 0.15 * np.arange(80))
    rows, off = (x.ravel(), y.ravel()), jittered(60, 80, 0.2, 15)
    other = P.PRISM_SCAN_BLOCKS if precision == P.PRISM_PRECISION_FP32 else P.PRISM_SCAN_TENSOR
    alone = []
    for pos, path in ((rows, P.PRISM_SCAN_ROWS), (off, other)):
        sim = plan(256, 16.0, 2, 15, precision=precision)
        base = held(sim)
        out = scan(sim, pos, 60, 80, path)
        alone.append((held(sim) - base, out))
        sim.close()
    sim = plan(256, 16.0, 2, 15, precision=precision)
    for _ in range(2):
        assert np.array_equal(scan(sim, rows, 60, 80, P.PRISM_SCAN_ROWS), alone[0][1])
        assert np.array_equal(scan(sim, off, 60, 80, other), alone[1][1])
    assert min(a for a, _ in alone) > 1 << 20
    assert held(sim) - base <= max(a for a, _ in alone) + (1 << 16)  # (counters)
    sim.close()


class SmallPool:
    """Device memory for the library's stream-ordered allocations up to `mb` megabytes (a multiple of 32, the
    grain of a pool), through a memory pool of that size in the place of the device's own."""

    class Props(ctypes.Structure):
        class Location(ctypes.Structure):
            _fields_ = [("type", ctypes.c_int), ("id", ctypes.c_int)]

        _fields_ = [("alloc", ctypes.c_int), ("handles", ctypes.c_int), ("location", Location), ("win32", ctypes.c_void_p),
                    ("max_size", ctypes.c_size_t), ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]

    def __init__(self, mb):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.mb = mb

    def __enter__(self):
        torch.cuda.synchronize()
        dev = torch.cuda.current_device()
        self.own, self.pool = ctypes.c_void_p(), ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.own), dev) == 0
        p = self.Props(1, 0, self.Props.Location(1, dev), None, self.mb << 20, 0)  # pinned device memory
        assert self.cu.cuMemPoolCreate(ctypes.byref(self.pool), ctypes.byref(p)) == 0
        assert self.cu.cuDeviceSetMemPool(dev, self.pool) == 0
        return self

    def __exit__(self, *exc):
        torch.cuda.synchronize()
        assert self.cu.cuDeviceSetMemPool(torch.cuda.current_device(), self.own) == 0
        assert self.cu.cuMemPoolDestroy(self.pool) == 0

    def most_used(self):
        v = ctypes.c_ulonglong()
        assert self.cu.cuMemPoolGetAttribute(self.pool, 8, ctypes.byref(v)) == 0  # CU_MEMPOOL_ATTR_USED_MEM_HIGH
        return v.value


@pytest.mark.parametrize("f,px,py,step,slack,path", [(4, 9, 125, 2.0, 4, P.PRISM_SCAN_LIST), (2, 4, 110, 0.5, 32, P.PRISM_SCAN_BLOCKS)])
def test_rows_without_memory_take_another_path(f, px, py, step, slack, path):
    # the rows' scratch does not fit beside the plan: the scan goes as positions off their rows would, and the
    # autotuner times what then runs
    x, y = np.meshgrid(step * np.arange(px), 0.14 * np.arange(py))
    pos = (x.ravel(), y.ravel())
    sim = plan(256, 16.0, f, 16)
    need = sim.info.device_bytes
    full = scan(sim, pos, px, py, P.PRISM_SCAN_ROWS)
    rows = P.prism_plan_info(sim.plan).device_bytes - need
    sim.close()
    mb = (need + (slack << 20) + (1 << 25) - 1) // (1 << 25) * 32
    assert need + rows > mb << 20
    with SmallPool(mb):
        sim = plan(256, 16.0, f, 16)
        out = scan(sim, pos, px, py, path)
        assert np.array_equal(scan(sim, pos, px, py, path), out)
        tuned = sim.autotune_scan(PROBE, *pos, DET, px=px, py=py).cpu().numpy()
        assert P.prism_plan_scan_path(sim.plan) == path and np.array_equal(tuned, out)
        ms = set(sim.tune_result()["scan"]["ms"].values())
        assert len(ms) == 1 if path == P.PRISM_SCAN_LIST else len(ms) > 1
        beams = sim.info.n_beams
        sim.close()
    close(out, full.astype(np.float64), beams)


def rows_cell(seed, precision=P.PRISM_PRECISION_FP32):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x, y = np.meshgrid(0.5 * np.arange(4), 0.14 * np.arange(110))
    return dict(grid=P.make_grid(256, 256, 1, 16.0, 16.0, 2.0, 300.0, 2, 2, 0.5, 20.0, precision=precision),
                V=50.0 * torch.rand((1, 256, 256), generator=g, device="cuda"), probe=PROBE, x0=x.ravel(), y0=y.ravel(), px=4, py=110, det=DET)


def run_batch(cells, budget=0):
    b = Batch(cells, hbm_budget_bytes=budget, n_branches=1)
    b.run()
    b.sync()
    out, held = [o.cpu().numpy() for o in b.outs], b.info.device_bytes
    b.close()
    return out, held


def least_bytes(cells):
    with pytest.raises(P.PrismError) as e:
        Batch(cells, hbm_budget_bytes=1)
    return int(re.search(r"batch needs (\d+) bytes", str(e.value)).group(1))


def test_a_batch_stays_within_its_budget_throughout():
    # the rows' scratch (some 120 MB a cell) is not allocated before the budget is looked at
    cells = [rows_cell(s) for s in (17, 18)]
    free, held = run_batch(cells)
    least = least_bytes(cells)
    assert held > least + (64 << 20)
    with SmallPool(4096) as pool:
        tight, used = run_batch(cells, least)
        assert used == least
        assert pool.most_used() <= least + (4 << 20)  # (allocations round up)
    for a, b in zip(tight, free):
        close(a, b.astype(np.float64), 213)


def test_rows_leave_later_cells_their_memory():
    # without a budget: the first cell's rows would leave no memory for the second cell's plan
    cells = [rows_cell(s) for s in (19, 20)]
    free, held = run_batch(cells)
    mb = (least_bytes(cells) + (40 << 20)) // (1 << 25) * 32
    assert held > mb << 20
    with SmallPool(mb):
        out, used = run_batch(cells)
    assert used <= mb << 20
    for a, b in zip(out, free):
        close(a, b.astype(np.float64), 213)


@pytest.mark.parametrize("n,cell,f,f_y,alpha,M,px,py,step", [
    (256, 16.0, 4, 2, 4.0, 0, 40, 9, 0.2),       # m = 0 alone, three beams along y; 32 x 64 windows
    (256, 16.0, 8, 4, 9.0, 0, 33, 5, 0.3),       # 16 x 32
    (256, 16.0, 4, 0, 5.0, 1, 41, 6, 0.2),       # one pair of m
    (256, 14.4, 2, 0, 25.0, 9, 12, 7, 0.3),      # 64 x 64, pairs of m in two chunks, three of them empty
    (256, 14.4, 2, 0, 36.0, 13, 9, 5, 0.2),      # in two chunks of 7
    (256, 16.0, 1, 0, 14.0, 11, 5, 6, 0.3),      # 128 x 128, two chunks
])
def test_rows_of_any_beam_set(n, cell, f, f_y, alpha, M, px, py, step):
    sim = plan(n, cell, f, 21, f_y=f_y, alpha=alpha)
    assert max(sim.beams()[0]) == M
    x, y = np.meshgrid(step * np.arange(px) - 1.3, step * np.arange(py) - 0.7)
    pos = (x.ravel(), y.ravel())
    out = scan(sim, pos, px, py, P.PRISM_SCAN_ROWS)
    some = np.array([0, px - 1, px * py // 2, px * py - 1])
    close(out[some], exact(sim, cell, f, f_y, pos[0][some], pos[1][some]), sim.info.n_beams)
    sim.close()


@pytest.mark.parametrize("n,cell,f", [(64, 8.0, 2), (256, 16.0, 4), (256, 12.5, 2)])
def test_small_value_and_remainder_rasters_by_rows(n, cell, f):
    sim = plan(n, cell, f, 22, precision=P.PRISM_PRECISION_FP16X2)
    x, y = np.meshgrid(0.3 * np.arange(4) - 0.5, 0.3 * np.arange(4) - 0.5)
    pos = (x.ravel(), y.ravel())
    out = scan(sim, pos, 4, 4, P.PRISM_SCAN_ROWS)
    ref = exact(sim, cell, f, 0, *pos)
    beams = sim.info.n_beams
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) <= 2.0 * (2.0 ** -20 * beams ** 0.5 + (beams + 24) * 2.0 ** -24)
    sim.close()


def test_wide_value_and_remainder_rasters_are_not_unpacked():
    # 32 x 32 probes 2 A apart reach the whole S-matrix (103 MB unpacked) for few windows on any part of it
    sim = plan(1024, 64.0, 16, 23, precision=P.PRISM_PRECISION_FP16X2)
    x, y = np.meshgrid(2.0 * np.arange(32), 2.0 * np.arange(32))
    scan(sim, (x.ravel(), y.ravel()), 32, 32, P.PRISM_SCAN_TENSOR)
    sim.close()


def test_parts_of_a_raster_agree_to_rounding():
    # a raster by rows against its bands of 6 rows (24 probes: a list), of whole rows that go by rows (bit for bit),
    # and its two left columns
    sim = plan(256, 16.0, 4, 24)
    beams = sim.info.n_beams
    x, y = np.meshgrid(0.2 * np.arange(4), 0.2 * np.arange(24))
    whole = scan(sim, (x.ravel(), y.ravel()), 4, 24, P.PRISM_SCAN_ROWS)
    for r in range(0, 24, 6):
        band = scan(sim, (x[r:r + 6].ravel(), y[r:r + 6].ravel()), 4, 6, P.PRISM_SCAN_LIST)
        close(band, whole[4 * r:4 * (r + 6)].astype(np.float64), beams)
    for r in range(0, 24, 8):
        band = scan(sim, (x[r:r + 8].ravel(), y[r:r + 8].ravel()), 4, 8, P.PRISM_SCAN_ROWS)
        assert np.array_equal(band, whole[4 * r:4 * (r + 8)])
    left = scan(sim, (x[:, :2].ravel(), y[:, :2].ravel()), 2, 24, P.PRISM_SCAN_LIST)
    close(left, whole.reshape(24, 4, -1)[:, :2].reshape(48, -1).astype(np.float64), beams)
    sim.close()
