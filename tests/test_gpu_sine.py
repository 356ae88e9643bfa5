"""Row transforms of the solves (sine.cuh: fold, three quarter-length FFTs) through the FP64 box
solve, whose rows use them, against scipy's DST for every line length (each pass plan: 4, 8, 8 x 2,
8 x 4, 8 x 8, 16 x 8, 16 x 16, 8 x 8 x 8), row counts that leave the last block partly filled, and
with and without box data."""
import numpy as np
import pytest
import scipy.fft as sf
import torch

import paper_2109_13628_gb300 as iim

pytestmark = pytest.mark.gpu


def reference(f, ring, nx, ny, h):
    f = f * (h * h)
    if ring is not None:
        f[0] += ring[1:nx]
        f[-1] += ring[nx + 2:2 * nx + 1]
        f[:, 0] += ring[2 * nx + 2:2 * nx + 1 + ny]
        f[:, -1] += ring[2 * nx + 1 + ny:]
    lx = 2 - 2 * np.cos(np.pi * np.arange(1, nx) / nx)
    ly = 2 - 2 * np.cos(np.pi * np.arange(1, ny) / ny)
    s = sf.dst(sf.dst(f, type=1, axis=1), type=1, axis=0) / (lx[None, :] + ly[:, None])
    return sf.dst(sf.dst(s, type=1, axis=1), type=1, axis=0) / (4 * nx * ny)


@pytest.mark.parametrize("nx,ny", [(16, 16), (32, 64), (64, 32), (128, 16), (256, 128), (512, 64), (1024, 32), (2048, 16)])
@pytest.mark.parametrize("ring", [False, True])
def test_row_transforms_through_the_box_solve(nx, ny, ring):
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(nx + ny)
    f = rng.normal(size=(ny - 1, nx - 1))
    r = rng.normal(size=2 * (nx + ny)) if ring else None
    h = 4.0 / nx
    T = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)
    u = torch.empty(ny - 1, nx - 1, dtype=torch.float64, device=dev)
    work = torch.empty(2 * (nx - 1) * (ny - 1), dtype=torch.float64, device=dev)
    iim.iim_box_poisson(iim.make_grid(0, 4, 0, h * ny, nx, ny), T(f), T(r) if ring else None, u, iim.IIM_FP64, work)
    ref = reference(f.copy(), r, nx, ny, h)
    # a few hundred rounding errors of 1e-16 at most; the column transforms of this call amplify theirs
    # by sqrt(ny)
    assert np.abs(u.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("nx,ny", [(16, 2048), (64, 1024), (1024, 512), (16, 256)])
def test_column_transforms_through_the_box_solve(nx, ny):
    """Column transforms at the line lengths whose result ends in either buffer (sine_ends_in_p)."""
    test_row_transforms_through_the_box_solve(nx, ny, True)
