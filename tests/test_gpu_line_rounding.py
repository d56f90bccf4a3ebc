"""The x lines in one exchange (32 x 16 and 32 x 32 points) round no worse than the staged lines of radices 8 8 8 and
8 16 8 that they stand in for: the same r2c of white noise with either, against float64.  Only the x lines differ, and
a transform's rounding does not depend on the run, so the comparison needs no margin."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [512, 1024])
def test_one_exchange_lines_round_no_worse(lib, n):
    from paper_1504_02591_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((n, n, n), generator=g, device="cuda")
    ref = torch.fft.rfftn(x.double())
    r = B.Recon(n, 5.0 * n, 1.6, 0.7, 15.0, (0.0, 0.0, 0.0), periodic=True, uniform=True)
    err = []
    for generic in (0, 1):
        r.set_option(B.OPT_KSPACE_GENERIC, generic)
        d = r.fft_r2c(x) - ref
        err.append(float(torch.linalg.vector_norm(torch.view_as_real(d)) / torch.linalg.vector_norm(torch.view_as_real(ref))))
        del d
    r.close()
    del x, ref
    torch.cuda.empty_cache()
    print(f"{n}^3 r2c of white noise: rel L2 error {err[0]:.4e} in one exchange, {err[1]:.4e} staged")
    assert err[0] <= err[1]
