"""Sweep paths of the pressure solve at the sizes where each can go wrong:
cluster-resident FP32 cycles, two-colour FP32 sweeps, FP32 rows that are no
multiple of 4 cells, and the chunked FP64 z lines."""
import numpy as np
import pytest

from paper_1511_07800_gb300 import inputs

from .conftest import gauge, rel_err
from .test_gpu_parity import case, schedule
from .test_gpu_zline import line_schedule, mean_free_rhs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 32, 32), (12, 16, 16), (8, 17, 33), (66, 10, 13), (30, 40, 16), (48, 32, 64)])
def test_cluster_cycles_bitwise(stp_lib, monkeypatch, shape):
    """A cycle on one cluster (variants 12 to 15: 16 or 8 blocks, slabs of
    levels or of rows) gives bitwise the launched sweeps (variant 0): same
    cell update, same values read.  Slabs of one to eight levels, uneven
    slabs, rows of 4-cell and of 2-cell vectors, two columns a thread."""
    nx, ny, nz = shape
    cfg = case(nx=nx, ny=ny, nz=nz, stretch=2.0)
    om = schedule(cfg, 32)
    b, _ = mean_free_rhs(cfg, 3)
    ref, ran = None, 0
    for v in (0, 12, 13, 14, 15):
        monkeypatch.setenv("STP_SWEEP_VARIANT", str(v))
        with stp_lib.Channel(cfg, precision="fp32", omega=om) as ch:
            p = np.zeros_like(b)
            st = ch.poisson_solve(b, p, tol=1e-8, maxit=96)
            took = ch.sweep_tile()[0]
        if ref is None:
            ref = (p, st["sweeps"])
        elif took == v:
            ran += 1
            assert st["sweeps"] == ref[1] and np.array_equal(p, ref[0]), v
    assert ran > 0


@pytest.mark.parametrize("shape,zline", [((128, 128, 130), 0), ((132, 128, 126), 0), ((134, 126, 126), 0),
                                         ((128, 128, 130), 1), ((132, 92, 192), 1), ((134, 170, 96), 1)])
def test_colour_solves_reach_the_tolerance(stp_lib, orc, monkeypatch, shape, zline):
    """Two-colour solves (at least 2^21 cells, even nx and ny) stop at
    ||b - L p|| <= 1e-8 ||b||, measured with the oracle's operator, and end at
    the Jacobi solves' pressure: both solve the same system to 1e-8, so they
    agree to the 1e-8 of the residual times the operator's conditioning on
    noise, far below 1e-5.  Half rows of whole float4, float2 and single
    entries; partial tiles; level counts of full and partial chunks.  The
    graph and the host-driven solve run the same kernels: bitwise."""
    nx, ny, nz = shape
    cfg = case(nx=nx, ny=ny, nz=nz, stretch=1.0, zline=zline)
    b, _ = mean_free_rhs(cfg, 5)
    got = []
    for colours, host in (("1", "0"), ("1", "1"), ("0", "0")):
        monkeypatch.setenv("STP_SRJ_COLOURS", colours)
        monkeypatch.setenv("STP_HOST_SOLVE", host)
        with stp_lib.Channel(cfg, precision="fp32") as ch:
            p = np.zeros_like(b)
            assert ch.poisson_solve(b, p, tol=1e-8)["converged"]
        got.append(p)
    r = b - orc.Oracle(dict(cfg, omega=[1.0])).laplacian(got[0])
    assert np.sqrt(np.sum(r * r) / np.sum(b * b)) <= 1e-8 * 1.0001
    assert np.array_equal(got[0], got[1])
    assert not np.array_equal(got[0], got[2])
    assert rel_err(got[0], got[2]) < 1e-5


@pytest.mark.parametrize("nz", [4, 47, 48, 49, 96, 97, 192, 193, 384, 385])
def test_line_f64_chunks(stp_lib, orc, nz):
    """FP64 z lines in chunks, at the edges of the chunk counts and levels (48,
    96, 192, 384) and just past the tallest, on partial column tiles: fixed
    sweeps against the oracle's Thomas solves to 1e-10."""
    cfg = case(nx=37, ny=4, nz=nz, stretch=2.0, zline=1)
    om = [0.6, 0.9, 0.7, 1.0]  # all below 2/mu_max: a contracting iteration
    cfg["omega"] = om
    b, rng = mean_free_rhs(cfg, 11)
    p0 = rng.standard_normal(b.shape) * 0.1
    p_o, it_o, _, _ = orc.Oracle(cfg).poisson(b, p0, tol=0.0, maxit=8)
    with stp_lib.Channel(cfg, omega=om) as ch:
        p_g = p0.copy()
        st = ch.poisson_solve(b, p_g, tol=0.0, maxit=8)
    assert st["sweeps"] == it_o == 8
    assert rel_err(p_g, gauge(p_o, cfg)) < 1e-10
