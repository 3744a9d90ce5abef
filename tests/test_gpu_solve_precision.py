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
    """An FP64 z-line cycle takes b - L p in differences of neighbours, which drop
    the pressure's level, so a solution stays where it is even under a large factor:
    two sweeps (20, then 0.5) from the solution itself move no cell by more than two
    units in its last place.  Half a unit each are the rounding of p once or
    twice (the second sweep amplifies nothing of the first's: |1 - mu/2| <= 1), of
    the mean and of the returned p - mean; 20 A^-1 times the rounding of the
    differences is some 1e-15, a hundredth of a unit.  Sweeps that form the line
    value of the pressure itself round with S p: 37 units at least."""
    cfg = inputs.preset("os_instability", nx=nx, ny=ny, nz=nz, stretch=stretch, zline=1)
    p0, b = offset_pressure(cfg)
    with stp_lib.Channel(cfg, precision="fp64", omega=[20.0, 0.5]) as ch:
        p = p0.copy()
        st = ch.poisson_solve(b, p, tol=0.0, maxit=2)
    assert st["sweeps"] == 2
    assert np.abs(p - gauge(p0, cfg)).max() <= 2 * 2.0 ** -43


def test_line_solve_to_a_tight_tolerance(stp_lib):
    """A strongly stretched channel (48 x 24 x 96, stretch 3) solved to 5e-12 of ||b||
    with z lines: the sweeps of a cycle run on a correction that keeps shrinking,
    and only its last addition rounds the pressure.  (Sweeps on the pressure stall
    at 8.7e-12 in residual form and at 1.5e-11 on line values.)"""
    cfg = inputs.preset("os_instability", nx=48, ny=24, nz=96, stretch=3.0, zline=1)
    p0, b = offset_pressure(cfg)
    with stp_lib.Channel(cfg, precision="fp64") as ch:
        p = np.zeros_like(p0)
        st = ch.poisson_solve(b, p, tol=5e-12, maxit=2048)
    assert st["converged"], st["rel_res"]


def fma(a, b, c):
    """a b + c with one rounding (the product is exact, or nearly, in long double)."""
    return (np.asarray(a, np.longdouble) * b + c).astype(np.float64)


def test_point_sweeps_round_as_little_as_ten_operations(stp_lib):
    """One cycle of FP64 point sweeps from the rounded solution leaves the residual of
    the sweeps' rounding.  It is at most a twelfth above that of the form
    p + omega ((sum c p_nb - b)/S - p) with fused multiplications, taken operation by
    operation here: partial sums of the same sizes are rounded either way, and 55
    thousand cells average them to a few per cent.  (The right-hand side added
    last: a seventh above.)"""
    nx, ny, nz = 48, 24, 48
    cfg = inputs.preset("os_instability", nx=nx, ny=ny, nz=nz, stretch=2.0)
    p0, b = offset_pressure(cfg)
    p0 = p0 - 700
    om, _, _ = stp_lib.srj_schedule(cfg)
    dz = np.diff(inputs.zfaces(cfg))
    zc = np.cumsum(dz) - 0.5 * dz
    hz = np.diff(zc)
    cup, cdn = np.zeros((nz, 1, 1)), np.zeros((nz, 1, 1))
    cup[:-1, 0, 0], cdn[1:, 0, 0] = 1 / (hz * dz[:-1]), 1 / (hz * dz[1:])
    idx2, idy2 = (nx / cfg["Lx"]) ** 2, (ny / cfg["Ly"]) ** 2
    iS = 1 / (2 * idx2 + 2 * idy2 + cup + cdn)

    def up(a):
        return np.concatenate([a[1:], a[-1:]])

    def down(a):
        return np.concatenate([a[:1], a[:-1]])

    def residual(p):
        lap = (idx2 * ((np.roll(p, -1, 2) - p) + (np.roll(p, 1, 2) - p)) +
               idy2 * ((np.roll(p, -1, 1) - p) + (np.roll(p, 1, 1) - p)) + cup * (up(p) - p) + cdn * (down(p) - p))
        return np.linalg.norm(b - lap) / np.linalg.norm(b)

    want = p0.copy()
    for w in om:
        nb = fma(idy2, np.roll(want, -1, 1) + np.roll(want, 1, 1), idx2 * (np.roll(want, -1, 2) + np.roll(want, 1, 2)))
        nb = fma(cdn, down(want), fma(cup, up(want), nb))
        want = fma(w, fma(nb - b, iS, -want), want)
    with stp_lib.Channel(cfg, precision="fp64") as ch:
        p = p0.copy()
        st = ch.poisson_solve(b, p, tol=0.0, maxit=len(om))
    assert st["sweeps"] == len(om)
    print("rounding of a cycle: residual %.3g, reference %.3g" % (residual(p), residual(want)))
    assert residual(p) <= 13 / 12 * residual(want)
