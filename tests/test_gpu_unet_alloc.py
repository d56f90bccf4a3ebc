"""The U-Net on grids that are refused: nothing is launched, and the network still works afterwards."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _net():
    from paper_1504_02591_gb300 import binding as B
    net = B.UNet(c1=8)
    rng = np.random.default_rng(3)
    net.set_params((0.1 * rng.standard_normal(net.get_params().size)).astype(np.float32))
    x = torch.from_numpy(rng.standard_normal((16, 16, 16, 5)).astype(np.float32)).cuda()
    return B, net, x


@pytest.mark.parametrize("n", [1296, 1624])
def test_grids_past_32bit_voxel_indices_are_refused(lib, n):
    """1296^3 is the first side of 2^31 voxels and more.  120 GB are held meanwhile, so that the activations
    of such a grid (219 GB) cannot be had either way; the refusal comes before anything is given back, so
    the last forward's layers are still there."""
    B, net, x = _net()
    y = net.forward(x)
    layer = net.get_layer(0, 16, 8)
    ballast = torch.empty(120 * 10 ** 9, dtype=torch.uint8, device="cuda")
    st = net.lib.recon_unet_forward(net.h, C.c_void_p(x.data_ptr()), n, C.c_void_p(y.data_ptr()))
    del ballast
    torch.cuda.empty_cache()
    assert st == B.ERR_OOM
    assert np.array_equal(net.get_layer(0, 16, 8), layer)
    net.close()


def test_forward_after_out_of_memory(lib):
    """A grid whose activations do not fit (c1 = 8, 1288^3: 223 GB, with 120 GB held) gives OOM; the next forward, on
    a side that had been allocated before, allocates again and gives the same output."""
    B, net, x = _net()
    y = net.forward(x)
    ballast = torch.empty(120 * 10 ** 9, dtype=torch.uint8, device="cuda")
    st = net.lib.recon_unet_forward(net.h, C.c_void_p(x.data_ptr()), 1288, C.c_void_p(y.data_ptr()))
    del ballast
    torch.cuda.empty_cache()
    assert st == B.ERR_OOM
    assert torch.equal(net.forward(x), y)
    net.close()
