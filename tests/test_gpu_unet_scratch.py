"""Device memory a network holds."""
import pytest

pytestmark = pytest.mark.gpu


def test_small_network_holds_no_more_than_its_parameters_need(stp_lib):
    """A network of 8 x 8 x 8 voxels has next to no activations: what it holds is its
    parameters with gradient and optimiser state (16 bytes each), their BF16 forms
    (wt, wtt and both in shared-memory order, 8 bytes and up to a third more in
    groups of 64 channels), and slices of the weight gradients for its few tiles
    (one slice a layer, 28 taps of 192 x 64 floats at most twice over): within 8 MB
    of that in all, allocations rounded up."""
    torch = pytest.importorskip("torch")
    first = stp_lib.UNet(1, 8, 8, 8)  # what the first network of a process loads
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    nets = [stp_lib.UNet(1, 8, 8, 8) for _ in range(4)]
    held = (before - torch.cuda.mem_get_info()[0]) / 4
    need = stp_lib.UNet.param_count() * (16 + 8 * 4 / 3)
    print("a network holds %.1f MB, its parameters need %.1f" % (held / 2 ** 20, need / 2 ** 20))
    assert held <= need + (8 << 20)
    for n in nets + [first]:
        n.close()
