"""Sine transforms with several lines per block (sine.cuh): 512- and 1024-point rows and columns, and a
small line length, at line counts beyond three full blocks per SM, none of them a multiple of the lines
per block, through the FP64 box solve against scipy's DST.

Bound: the solve's eigenvalues are 2 - 2 cos, each cosine within a rounding error of 2^-53, so the lowest
mode carries a relative error of up to 8 2^-53 / (lx + ly); the transforms themselves stay below 1e-12."""
import numpy as np
import pytest
import scipy.fft as sf
import torch

import paper_2109_13628_gb300 as iim

pytestmark = pytest.mark.gpu


# (nx, ny, lines per block of the rows or columns): rows have ny - 1 lines of nx points, columns nx of ny
@pytest.mark.parametrize("nx,ny,per_row,per_col", [(512, 2048, 4, 1), (2048, 512, 1, 4), (1024, 1024, 2, 2), (16, 2048, 4, 1)])
def test_several_lines_per_block(nx, ny, per_row, per_col):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for lines, per in ((ny - 1, per_row), (nx, per_col)):
        assert per == 1 or (lines >= 3 * sms * per), "this device does not reach the form"
    rng = np.random.default_rng(nx + ny)
    f = rng.normal(size=(ny - 1, nx - 1))
    h = 4.0 / nx
    T = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    u = torch.empty(ny - 1, nx - 1, dtype=torch.float64, device="cuda")
    work = torch.empty(2 * (nx - 1) * (ny - 1), dtype=torch.float64, device="cuda")
    iim.iim_box_poisson(iim.make_grid(0, 4, 0, h * ny, nx, ny), T(f), None, u, iim.IIM_FP64, work)
    lx, ly = (4 * np.sin(np.pi * np.arange(1, n) / (2 * n)) ** 2 for n in (nx, ny))
    s = sf.dst(sf.dst(f * h * h, type=1, axis=1), type=1, axis=0) / (lx[None, :] + ly[:, None])
    ref = sf.dst(sf.dst(s, type=1, axis=1), type=1, axis=0) / (4 * nx * ny)
    bound = 8 * 2.0 ** -53 / (lx[0] + ly[0]) + 1e-12
    assert np.abs(u.cpu().numpy() - ref).max() <= bound * np.abs(ref).max()
