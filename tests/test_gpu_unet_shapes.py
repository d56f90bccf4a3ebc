"""The U-Net's gradients at grid sides whose levels do not fill the kernels' tiles (4 x 4 x 32 voxels, 256- and
512-voxel blocks), for both widths and both storage types, against the FP64 oracle.

float32 storage: sums of at most 96 x 27 products forward and 24^3 voxels backward, each rounding 6e-8
in quadrature through 11 layers both ways: 6e-8 sqrt(2600 x 22) = 1.4e-5 of the summed magnitudes; the bound
leaves the factor of ten that cancelling gradients need.  bfloat16 storage rounds every activation by
2^-9 = 2e-3; gradients through ten such layers are held to ten times that in the L2 norm.
"""
import numpy as np
import pytest

from oracle import unet_oracle as U

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / max((b ** 2).sum(), 1e-300)))


@pytest.mark.parametrize("n,c1,bf16", [(8, 16, False), (24, 8, False), (40, 8, False), (16, 16, True), (24, 8, True)])
def test_gradients_at_ragged_sides(lib, n, c1, bf16):
    from paper_1504_02591_gb300 import binding as B
    rng = np.random.default_rng(n + c1)
    params = U.init_params(n, c1=c1)
    params["head"] = (rng.standard_normal((1, c1, 1)) * 0.3, np.array([0.05]))
    for k in params:
        w, b = params[k]
        params[k] = (w, b + 0.05 * rng.standard_normal(b.shape))
    specs = U.layer_specs(c1)
    net = B.UNet(c1=c1, bf16=bf16)
    flat = B.flat_params(params, specs)
    net.set_params(flat)
    p32 = B.unflat_params(flat.astype(np.float64), specs)
    x = rng.standard_normal((n, n, n, 5)).astype(np.float32)
    t = rng.standard_normal((n, n, n)).astype(np.float32)
    y = net.forward(torch.from_numpy(x)).cpu().numpy()
    y_ref, _ = U.forward(p32, x.astype(np.float64))
    loss = net.backward(torch.from_numpy(x), torch.from_numpy(t))
    L_ref, g_ref = U.backward(p32, x.astype(np.float64), t.astype(np.float64)[..., None])
    tol = 2e-2 if bf16 else 1.4e-4
    assert _rel(y, y_ref[..., 0]) < tol
    assert loss == pytest.approx(L_ref, rel=tol)
    g = B.unflat_params(net.get_grads().astype(np.float64), specs)
    if bf16:
        a = np.concatenate([np.ravel(v) for k, _, _ in specs for v in g[k]])
        b = np.concatenate([np.ravel(v) for k, _, _ in specs for v in g_ref[k]])
        assert _rel(a, b) < tol
    else:
        for name, _, _ in specs:
            assert _rel(g[name][0], g_ref[name][0]) < tol, name
            assert _rel(g[name][1], g_ref[name][1]) < tol, name
    net.close()
