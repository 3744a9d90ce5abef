"""Kernel variants of the U-Net at the sizes where each can go wrong: tcgen05
blocks that stay for several tiles, and layers of tiny and ragged levels."""
import numpy as np
import pytest

from .test_gpu_unet import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 32, 64, 128), (3, 8, 80, 72), (2, 8, 16, 304)])
def test_tcgen05_blocks_of_many_tiles(stp_lib, orc, monkeypatch, shape):
    """Full-resolution layers of 512 to 2048 tiles of 8 x 16 x 1 voxels: blocks
    that take several tiles and others that take one fewer, both halo and
    accumulator stages in turn, resident and streamed weights, tiles of 4, 2
    and 1 planes.  Every accumulator sees the same MMAs in the same order, so
    the forward output is bitwise the same however the tiles are cut."""
    torch = pytest.importorskip("torch")
    unet, theta, x, _ = _setup(6, shape)
    n, d, h, w = x.shape
    tx = torch.from_numpy(x.astype(np.float32)).cuda()
    got = []
    for planes in ("1", "2", "4", "0"):
        monkeypatch.setenv("STP_UNET_TC_PLANES", planes)
        net = stp_lib.UNet(n, d, h, w)
        net.set_params(theta.astype(np.float32))
        ty = torch.zeros_like(tx)
        net.forward(tx, ty)
        got.append(ty.cpu().numpy())
        net.close()
    for g in got[1:]:
        assert np.array_equal(g, got[0])


@pytest.mark.parametrize("shape", [(1, 8, 8, 8), (2, 8, 24, 40), (1, 24, 8, 56), (3, 16, 16, 8)])
def test_tiny_and_ragged_levels(stp_lib, orc, shape):
    """Levels down to 1 x 1 x 1 and 1 x 3 x 5 voxels, batches of 1 to 3, widths
    that leave partial tiles in each direction: forward and gradient against
    the oracle with its storage points rounded to bfloat16, within the bounds
    of the regular shapes (FP32 order, and a rounding of a stored value where
    the orders straddle one)."""
    torch = pytest.importorskip("torch")
    unet, theta, x, t = _setup(7, shape)
    n, d, h, w = x.shape
    net = stp_lib.UNet(n, d, h, w)
    net.set_params(theta.astype(np.float32))
    tx = torch.from_numpy(x.astype(np.float32)).cuda()
    tt = torch.from_numpy(t.astype(np.float32)).cuda()
    ty = torch.zeros_like(tx)
    net.forward(tx, ty)
    y = ty.cpu().numpy().astype(np.float64)
    y_b = unet.forward(theta, x[..., None], rnd=unet.bf16)[..., 0]
    assert np.abs(y - y_b).max() < 2e-2 * np.abs(y_b).max()
    g = torch.zeros(stp_lib.UNet.param_count(), dtype=torch.float32, device="cuda")
    loss = net.gradient(tx, tt, g)
    L_o, g_o = unet.loss_and_grad(theta, x[..., None], t[..., None], rnd=unet.bf16)
    gg = g.cpu().numpy().astype(np.float64)
    assert abs(loss - L_o) < 1e-2 * L_o
    rel = np.linalg.norm(gg - g_o) / np.linalg.norm(g_o)
    assert rel < 5e-2, rel
    net.close()


@pytest.mark.parametrize("shape", [(1, 8, 128, 64), (2, 16, 128, 64)])
def test_streamed_weights_of_the_deepest_level(stp_lib, orc, monkeypatch, shape):
    """A network whose 128-channel level runs on tcgen05 too (16 rows): weights
    of 64 to 128 and 128 to 128 channels through the ring, two groups of
    channels, one and two planes a level.  Against the mma.sync kernels within
    the bounds of the smaller shapes."""
    torch = pytest.importorskip("torch")
    unet, theta, x, t = _setup(8, shape)
    n, d, h, w = x.shape
    tx = torch.from_numpy(x.astype(np.float32)).cuda()
    tt = torch.from_numpy(t.astype(np.float32)).cuda()
    out = []
    for tc in ("0", "1"):
        monkeypatch.setenv("STP_UNET_TC", tc)
        net = stp_lib.UNet(n, d, h, w)
        net.set_params(theta.astype(np.float32))
        ty = torch.zeros_like(tx)
        net.forward(tx, ty)
        g = torch.zeros(stp_lib.UNet.param_count(), dtype=torch.float32, device="cuda")
        net.gradient(tx, tt, g)
        out.append((ty.cpu().numpy().astype(np.float64), g.cpu().numpy().astype(np.float64)))
        net.close()
    (y0, g0), (y1, g1) = out
    assert np.abs(y1 - y0).max() < 2e-2 * np.abs(y0).max()
    assert np.linalg.norm(g1 - g0) < 5e-2 * np.linalg.norm(g0)
