"""Multislice detector lists and probe apertures made for the device: against the fixed-scratch entry point,
which makes them on the host from the same definitions (bitwise), at odd detectors and apertures."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1702_01904_gb300 import prism as P  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,cx,cy", [(16, 16, 4.0, 4.0), (64, 32, 8.0, 5.1), (32, 128, 3.7, 9.0), (256, 256, 16.0, 16.0)])
@pytest.mark.parametrize("det", [(0.0, 1.0, 100), (0.0, 1.0e4, 1), (7.3, 0.11, 4096), (-50.0, 3.7, 77), (1.0e5, 1.0, 5)])
@pytest.mark.parametrize("probe", [(20.0, 0.0, 0.0), (0.0, 3.0e-2, 0.0), (500.0, 0.0, 0.0), (12.0, -0.2, 0.35)])
def test_lists_and_apertures_equal_the_host_ones(nx, ny, cx, cy, det, probe):
    # runs of one pixel, bins past the grid, a negative start, empty lists; apertures of one pixel, wider than
    # the grid, tilted across its edge
    g = P.make_grid(nx, ny, 2, cx, cy, 2.0, 300.0, 1, 1, 0.5, 20.0)
    V = torch.rand((2, ny, nx), generator=torch.Generator().manual_seed(3)).mul_(60.0).cuda()
    x0 = np.array([0.1, cx * 0.7, -1.3])
    y0 = np.array([0.2, cy * 0.4, 2.0 * cy])
    pr = P.make_probe(probe[0], 10.0, 0.0, probe[1], probe[2])
    d = P.make_detector(*det)
    a = torch.full((3, det[2]), 7.0, device="cuda")
    b = torch.full((3, det[2]), 8.0, device="cuda")
    sc = P.make_scan(3, 1, x0, y0)
    s = torch.cuda.current_stream()
    P.multislice_scan_run(g, V, pr, sc, d, a, s)
    P.multislice_scan_run_noalloc(g, V, pr, sc, d, b, s)
    torch.cuda.synchronize()
    assert torch.equal(torch.nan_to_num(a, nan=-1.0), torch.nan_to_num(b, nan=-1.0))
