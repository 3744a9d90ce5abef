"""How FP64 pressure sweeps round."""
import numpy as np
import pytest

from paper_1511_07800_gb300 import inputs

from .conftest import gauge

pytestmark = pytest.mark.gpu


def offset_pressure(cfg):
    """A smooth pressure between 512 and 1024 (so that its last place is 2^-43),
    and b = L p of exactly these values, in long double, rounded to FP64."""
    ld = np.longdouble
    nx, ny, nz = cfg["nx"], cfg["ny"], cfg["nz"]
    zf = inputs.zfaces(cfg).astype(ld)
    dz, zc = np.diff(zf), 0.5 * (zf[1:] + zf[:-1])
    hz, w = np.diff(zc)[:, None, None], dz[:, None, None]
    x = (np.arange(nx) * 2 * np.pi / nx)[None, None, :]
    y = (np.arange(ny) * 2 * np.pi / ny)[None, :, None]
    z = (zc / cfg["Lz"] * np.pi).astype(np.float64)[:, None, None]
    p = 700 + np.cos(x) * np.sin(y) * np.cos(z) + 0.5 * np.sin(x) * np.cos(2 * z)
    a = p.astype(ld)
    fz = np.zeros((nz + 1, ny, nx), ld)
    fz[1:-1] = (a[1:] - a[:-1]) / hz
    b = ((np.roll(a, -1, 2) - 2 * a + np.roll(a, 1, 2)) * (nx / ld(cfg["Lx"])) ** 2 +
         (np.roll(a, -1, 1) - 2 * a + np.roll(a, 1, 1)) * (ny / ld(cfg["Ly"])) ** 2 + (fz[1:] - fz[:-1]) / w)
    return p, (b - np.sum(b * w) / (np.sum(w) * nx * ny)).astype(np.float64)


@pytest.mark.parametrize("nx,ny,nz,stretch", [(32, 16, 32, 0.0), (48, 24, 48, 2.0), (37, 21, 66, 2.0), (64, 32, 97, 2.0),
                                              (16, 8, 200, 2.0)])
def test_line_sweeps_round_with_the_differences(stp_lib, nx, ny, nz, stretch):
    """An FP64 z-line sweep forms b - L p in differences of neighbours, which drop
    the pressure's level, so a solution stays where it is even under a large factor:
    two sweeps (20, then 0.5) from the solution itself move no cell by more than two
    units in its last place.  Half a unit is each sweep's rounding of p (the
    second sweep amplifies none of the first's: |1 - mu/2| <= 1) and half each the
    rounding of the mean and of the returned p - mean; 20 A^-1 times the rounding of
    the differences is some 1e-15, a hundredth of a unit.  Sweeps that form the
    line value itself round with S p: 37 units at least."""
    cfg = inputs.preset("os_instability", nx=nx, ny=ny, nz=nz, stretch=stretch, zline=1)
    p0, b = offset_pressure(cfg)
    with stp_lib.Channel(cfg, precision="fp64", omega=[20.0, 0.5]) as ch:
        p = p0.copy()
        st = ch.poisson_solve(b, p, tol=0.0, maxit=2)
    assert st["sweeps"] == 2
    assert np.abs(p - gauge(p0, cfg)).max() <= 2 * 2.0 ** -43
