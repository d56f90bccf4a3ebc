"""A workspace short of the register-fused kernels' fourth vector field (the size that was enough before the
384 and 1024 meshes had those kernels, and less) still gives a handle: it runs the generic kernels."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [256, 384])
def test_workspace_without_the_fourth_field(lib, n):
    from paper_1504_02591_gb300 import binding as B
    L = 5.0 * n
    args = (n, L, 1.6, 0.7, 15.0, (-0.3 * L, 0.5 * L, 0.4 * L))
    g = torch.Generator(device="cuda").manual_seed(n)
    gal = torch.rand((200_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    r = B.Recon(*args, periodic=True, uniform=True)
    field = 4 * n ** 3 + 8 * n * n
    out = {}
    for what, missing in (("whole", 0), ("small", field)):
        r.close()
        r.ws_bytes = r.workspace.numel() - missing
        h = C.c_void_p()
        st = r.lib.recon_create(C.byref(r.params), C.c_void_p(r.stream.cuda_stream), C.c_void_p(r.workspace.data_ptr()),
                                r.ws_bytes, C.byref(h))
        assert st == B.OK
        r.h = h
        guard = r.workspace[r.ws_bytes:].fill_(77)
        for plane in (0, 16):                        # accepted, and without effect on the generic kernels
            r.set_option(B.OPT_PLANE_BATCH, plane)
            r.deposit(gal)
            r.smooth()
            r.start_features(B.START_FFTA, 1)
            r.deposit(gal)
            r.smooth()
            r.iterate(B.START_FFTA, 0.0, 3)
            out[what] = (r.get_psi(), r.shift(gal, True))
        assert bool((guard == 77).all())
    for a, b in zip(out["whole"], out["small"]):
        assert float((a - b).norm() / a.norm()) < 2e-6   # float32 rounding of the transforms, 3e-7 each
    r.close()
    h = C.c_void_p()
    assert r.lib.recon_create(C.byref(r.params), C.c_void_p(r.stream.cuda_stream), C.c_void_p(r.workspace.data_ptr()),
                              r.workspace.numel() - field - 256, C.byref(h)) == B.ERR_OOM
