"""Which kernels a pressure solve runs, and what must not depend on that choice."""
import numpy as np
import pytest

from .conftest import gauge, rel_err
from .test_gpu_parity import case, schedule, turbulent_like
from .test_gpu_zline import mean_free_rhs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,zline", [((128, 128, 130), 0), ((132, 128, 126), 0), ((134, 126, 126), 0),
                                         ((256, 128, 65), 1), ((256, 92, 96), 1), ((252, 90, 97), 1),
                                         ((134, 170, 96), 1), ((128, 128, 192), 1)])
def test_colour_variants_bitwise(stp_lib, monkeypatch, shape, zline):
    """The tile shapes among which a two-colour sweep is picked by timing give the
    same bits (two cycles from zero), so that a resumed run does not depend on
    the clock: half rows of whole float4, float2 and single entries, z lines in
    16 and in 32 level chunks, full and partial."""
    nx, ny, nz = shape
    cfg = case(nx=nx, ny=ny, nz=nz, stretch=1.0, zline=zline)
    b, _ = mean_free_rhs(cfg, 5)
    M = len(stp_lib.srj_schedule(cfg)[0])
    ran = {}
    for v in (0, 1, 2):
        monkeypatch.setenv("STP_COLOUR_VARIANT", str(v))
        with stp_lib.Channel(cfg, precision="fp32") as ch:
            p = np.zeros_like(b)
            ch.poisson_solve(b, p, tol=0.0, maxit=2 * M)
            ran[ch.sweep_tile()[0]] = p
    # rows that hold no whole vectors of a width leave it out
    widths = [w for w in (4, 2, 1) if nx // 2 % w == 0]
    assert sorted(ran) == ([0, 1, 2][-len(widths):] if zline else [0, 1, 2])
    first = ran[min(ran)]
    for v, p in ran.items():
        assert np.array_equal(p, first), v


@pytest.mark.parametrize("shape,zline,jacobi", [((134, 170, 96), 1, True), ((128, 128, 130), 1, True),
                                                ((128, 128, 130), 0, False)])
def test_line_variant_0_keeps_jacobi_sweeps(stp_lib, monkeypatch, shape, zline, jacobi):
    """STP_LINE_VARIANT=0 keeps Jacobi sweeps on every z-line grid, also one whose
    rows are no multiple of 32 cells: bitwise those of STP_SRJ_COLOURS=0.  It says
    nothing about point sweeps."""
    nx, ny, nz = shape
    cfg = case(nx=nx, ny=ny, nz=nz, stretch=1.0, zline=zline)
    b, _ = mean_free_rhs(cfg, 5)
    M = len(stp_lib.srj_schedule(cfg)[0])
    monkeypatch.setenv("STP_LINE_VARIANT", "0")
    got = []
    for colours in ("1", "0"):
        monkeypatch.setenv("STP_SRJ_COLOURS", colours)
        with stp_lib.Channel(cfg, precision="fp32") as ch:
            p = np.zeros_like(b)
            ch.poisson_solve(b, p, tol=0.0, maxit=M)
        got.append(p)
    assert np.array_equal(*got) == jacobi


@pytest.mark.parametrize("shape,zline,precision,env,want", [
    ((128, 128, 130), 0, "fp32", {}, "k_col_point"),
    ((134, 170, 96), 1, "fp32", {}, "k_col_line"),
    ((134, 170, 96), 1, "fp32", {"STP_LINE_VARIANT": "0"}, "k_line_sweep_smem"),
    ((128, 128, 130), 1, "fp32", {"STP_LINE_VARIANT": "0"}, "k_line_sweep_vec"),
    ((128, 128, 130), 0, "fp32", {"STP_LINE_VARIANT": "0"}, "k_col_point"),
    ((128, 128, 130), 1, "fp32", {"STP_SRJ_COLOURS": "0"}, "k_line_sweep_chunk"),
    ((8, 5, 800), 1, "fp32", {}, "k_line_sweep<float>"),
    ((64, 24, 32), 1, "fp32", {"STP_LINE_PERSISTENT": "1"}, "k_line_cycle_f32"),
    ((64, 24, 32), 0, "fp32", {"STP_PERSISTENT": "1"}, "k_cycle_f32"),
    ((32, 32, 32), 0, "fp32", {"STP_SWEEP_VARIANT": "12"}, "k_cluster_cycle"),
    ((64, 24, 32), 0, "fp32", {"STP_SWEEP_VARIANT": "4"}, "k_sweep_f32_z<4,4>"),
    ((64, 24, 32), 0, "fp32", {"STP_SWEEP_VARIANT": "10"}, "k_sweep_f32_pair<4,4>"),
    ((37, 24, 32), 0, "fp32", {}, "k_sweep_f32<1>"),
    ((64, 24, 32), 0, "fp64", {}, "k_sweep_f64"),
    ((64, 24, 32), 1, "fp64", {}, "k_line_f64"),
    ((8, 5, 400), 1, "fp64", {}, "k_line_sweep<double>"),
])
def test_sweep_kernel_names_what_runs(stp_lib, monkeypatch, shape, zline, precision, env, want):
    """stp_sweep_kernel follows the dispatch of the solve."""
    nx, ny, nz = shape
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    cfg = case(nx=nx, ny=ny, nz=nz, stretch=1.0, zline=zline)
    b, _ = mean_free_rhs(cfg, 5)
    with stp_lib.Channel(cfg, precision=precision) as ch:
        ch.poisson_solve(b, np.zeros_like(b), tol=0.0, maxit=32)
        assert ch.sweep_kernel() == want


@pytest.mark.parametrize("order", ["short first", "long first", "persistent first"])
def test_tile_choice_is_per_cycle_length(stp_lib, monkeypatch, order):
    """What the autotuner picks for one handle says nothing about a handle of
    another cycle length, or without persistent cycles, on the same grid: a cluster
    loads and stores its channel once a cycle, far too often for cycles of two
    sweeps and well worth it for long ones (32 x 32 x 32: 0.7 of the best
    launched sweep)."""
    # grids of their own: choices are kept for the process
    cfg = case(nx=32, ny=32, nz={"short first": 33, "long first": 34, "persistent first": 36}[order], stretch=0.0)
    b, _ = mean_free_rhs(cfg, 5)

    def kernel(omega=None):
        with stp_lib.Channel(cfg, precision="fp32", omega=omega) as ch:
            ch.poisson_solve(b, np.zeros_like(b), tol=0.0, maxit=2)
            return ch.sweep_kernel()

    short = [1.0, 1.0]
    if order == "long first":
        assert kernel() == "k_cluster_cycle"
        assert kernel(short).startswith("k_sweep_f32")
        return
    if order == "short first":
        assert kernel(short).startswith("k_sweep_f32")
    else:
        monkeypatch.setenv("STP_PERSISTENT", "1")
        assert kernel() == "k_cycle_f32"
        monkeypatch.delenv("STP_PERSISTENT")
    assert kernel() == "k_cluster_cycle"


CLUSTER_COLUMNS = [
    # shape, variants it fits, those among them of two columns a thread
    ((76, 57, 32), {12, 13}, {12}),              # 4-cell vectors, slabs of 2 levels; 1083 columns
    ((76, 32, 57), {12, 13}, {13}),              # the same across y
    ((76, 27, 48), {12, 13, 14, 15}, {14}),      # slabs of up to 6 on 8 blocks, 513 columns of 512 threads
    ((76, 48, 27), {12, 13, 14, 15}, {15}),
    ((76, 40, 96), {12}, {12}),                  # slabs of 6 on 16 blocks, 760 columns
    ((76, 96, 27), {13}, {13}),
    ((66, 33, 32), {12, 13, 14}, {12, 13, 14}),  # 2-cell vectors, slabs of 2 and of 4, odd column counts
    ((66, 32, 33), {12, 13, 15}, {12, 13, 15}),
    ((76, 57, 16), {12, 13, 14, 15}, {12, 14}),  # slabs of one level
]


@pytest.mark.parametrize("shape,fits,two", CLUSTER_COLUMNS)
def test_cluster_two_columns_a_thread_bitwise(stp_lib, monkeypatch, shape, fits, two):
    """Cluster-resident cycles whose blocks have more columns than threads, so that
    a thread takes two: bitwise the launched sweeps, and every variant that fits
    did run."""
    nx, ny, nz = shape
    assert two <= fits
    cfg = case(nx=nx, ny=ny, nz=nz, stretch=2.0)
    om = schedule(cfg, 32)
    b, _ = mean_free_rhs(cfg, 3)
    ref, ran = None, set()
    for v in (0, 12, 13, 14, 15):
        monkeypatch.setenv("STP_SWEEP_VARIANT", str(v))
        with stp_lib.Channel(cfg, precision="fp32", omega=om) as ch:
            p = np.zeros_like(b)
            st = ch.poisson_solve(b, p, tol=1e-8, maxit=96)
            if ch.sweep_kernel() == "k_cluster_cycle":
                ran.add(ch.sweep_tile()[0])
        if ref is None:
            ref = (p, st["sweeps"])
        assert st["sweeps"] == ref[1] and np.array_equal(p, ref[0]), v
    assert ran == fits


def test_sweeps_without_a_table(stp_lib, orc):
    """FP64 point sweeps whose level coefficients would exceed the table's 80 MB (4096
    sweeps a cycle, 430 levels: 85 MB) form them in the kernel: a cycle of
    contracting factors against the oracle to 1e-10."""
    cfg = case(nx=6, ny=5, nz=430, stretch=2.0)
    om = [0.6, 0.9, 0.7, 1.0] * 1024
    cfg["omega"] = om
    b, rng = mean_free_rhs(cfg, 11)
    p0 = rng.standard_normal(b.shape) * 0.1
    p_o, it_o, _, _ = orc.Oracle(cfg).poisson(b, p0, tol=0.0, maxit=4096)
    with stp_lib.Channel(cfg, omega=om) as ch:
        p_g = p0.copy()
        st = ch.poisson_solve(b, p_g, tol=0.0, maxit=4096)
    assert st["sweeps"] == it_o == 4096
    assert rel_err(p_g, gauge(p_o, cfg)) < 1e-10


@pytest.mark.parametrize("zline,host", [(0, "0"), (1, "0"), (0, "1")])
def test_network_on_and_off_a_two_colour_channel(stp_lib, orc, monkeypatch, zline, host):
    """A learned guess takes a large channel from two-colour to Jacobi sweeps and
    back: layout of the residual and the correction, tile choice and solve graph
    all change.  With the network (as the guess and as the preconditioner) solves
    reach 1e-8 measured with the oracle's operator; without it again they end
    bitwise where they did before."""
    unet = pytest.importorskip("oracle.unet")
    monkeypatch.setenv("STP_HOST_SOLVE", host)
    n = 128
    cfg = case(nx=n, ny=n, nz=n, stretch=0.0, zline=zline)
    b, _ = mean_free_rhs(cfg, 5)
    oracle = orc.Oracle(dict(cfg, omega=[1.0]))
    colour = "k_col_line" if zline else "k_col_point"
    net = stp_lib.UNet(1, n, n, n)
    net.set_params(unet.init_params(11).astype(np.float32))
    net.set_output_scale(1e3)  # an untrained network: small corrections
    with stp_lib.Channel(cfg, precision="fp32") as ch:

        def solve():
            p = np.zeros_like(b)
            st = ch.poisson_solve(b, p, tol=1e-8)
            r = b - oracle.laplacian(p)
            assert st["converged"] and np.sqrt(np.sum(r * r) / np.sum(b * b)) <= 1e-8 * 1.0001
            return p

        first = solve()
        assert ch.sweep_kernel() == colour
        for mode in (0, 1):
            ch.set_learned_mode(mode)
            ch.set_learned_guess(net)
            solve()
            assert ch.sweep_kernel() not in ("", colour)
        ch.set_learned_guess(None)
        again = solve()
        assert ch.sweep_kernel() == colour
        assert np.array_equal(again, first)
    net.close()


def test_two_colour_channel_in_a_batch(stp_lib):
    """Channels of two-colour sweeps, point and z line, beside channels that are
    solved in a group: each ends bitwise where it ends when stepped alone."""
    specs = [case(nx=128, ny=128, nz=128, nu=1 / 500.0),
             case(nx=32, ny=16, nz=32, nu=1 / 500.0),
             case(nx=160, ny=116, nz=114, nu=1 / 500.0, stretch=1.0, zline=1),
             case(nx=32, ny=16, nz=32, nu=1 / 800.0)]
    alone, kernels = [], []
    for i, cfg in enumerate(specs):
        with stp_lib.Channel(cfg, precision="fp32") as ch:
            ch.set_fields(*turbulent_like(cfg, 30 + i))
            ch.step(2)
            alone.append(ch.get_fields())
            kernels.append(ch.sweep_kernel())
    assert kernels[0] == "k_col_point" and kernels[2] == "k_col_line"
    chans = [stp_lib.Channel(cfg, precision="fp32") for cfg in specs]
    for i, ch in enumerate(chans):
        ch.set_fields(*turbulent_like(specs[i], 30 + i))
    batch = stp_lib.Batch(chans)
    st = batch.step(2)
    assert st["converged"]
    assert [g["channels"] for g in batch.groups()] == [2]
    for i, ch in enumerate(chans):
        got = ch.get_fields()
        for k in ("u", "v", "w", "p"):
            assert np.array_equal(got[k], alone[i][k]), (i, k)
    batch.close()
    for ch in chans:
        ch.close()


def test_line_f64_cycles_wherever_they_run(stp_lib, monkeypatch):
    """FP64 z-line cycles borrow arrays of the velocity half step for the residual
    and the correction: whole steps by the solve graph, driven from the host, and in
    a batch beside a second channel end bitwise alike."""
    specs = [case(nx=37, ny=12, nz=50, stretch=2.0, zline=1, les=1, nu=1 / 500.0),
             case(nx=32, ny=16, nz=20, nu=1 / 500.0, zline=1, cn_zline=1)]
    alone = []
    for host in ("0", "1"):
        monkeypatch.setenv("STP_HOST_SOLVE", host)
        for i, cfg in enumerate(specs):
            with stp_lib.Channel(cfg, precision="fp64") as ch:
                ch.set_fields(*turbulent_like(cfg, 40 + i))
                assert ch.step(4)["converged"]
                assert ch.sweep_kernel() == "k_line_f64"
                alone.append(ch.get_fields())
    monkeypatch.delenv("STP_HOST_SOLVE")
    chans = [stp_lib.Channel(cfg, precision="fp64") for cfg in specs]
    for i, ch in enumerate(chans):
        ch.set_fields(*turbulent_like(specs[i], 40 + i))
    batch = stp_lib.Batch(chans)
    assert batch.step(4)["converged"]
    for i, ch in enumerate(chans):
        got = ch.get_fields()
        for k in ("u", "v", "w", "p"):
            assert np.array_equal(got[k], alone[i][k]) and np.array_equal(alone[2 + i][k], alone[i][k]), (i, k)
    batch.close()
    for ch in chans:
        ch.close()
