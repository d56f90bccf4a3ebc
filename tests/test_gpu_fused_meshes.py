"""The register-fused passes against the staged generic ones (RECON_OPT_KSPACE_GENERIC) on every mesh side
that has both: the analytic starts, both lines of sight, both x-line tiles, y-plane batches, and the
warm start's radial, upsampling and supplied-displacement passes.

Tolerance: both are float32 transforms of 3 log2 N radix-2 levels, each level adding at most one rounding
(6e-8) in quadrature per pass of an update; with N <= 1024 that is 6e-8 sqrt(30) = 3.3e-7 per 3-D
transform and, for two independent sides and the two transforms of an update, 6.6e-7 in the L2 norm.
The bound is three times that.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-6


def _box(n, los, seed=5):
    from paper_1504_02591_gb300 import binding as B
    L = 6.84 * n
    obs = (0.48, -0.6, 0.64) if los else (-0.8 * L, 0.45 * L, 0.6 * L)
    r = B.Recon(n, L, 1.7, 0.75, 15.0, obs, B.LOS_FIXED if los else B.LOS_RADIAL, True, 0.01, False, True)
    g = torch.Generator(device="cuda").manual_seed(seed)
    # clustered tracers: uniform points and a Gaussian clump round each of 64 centres
    c = torch.rand((64, 3), generator=g, device="cuda", dtype=torch.float64) * L
    p = c.repeat_interleave(4000, 0) + 30.0 * torch.randn((256_000, 3), generator=g, device="cuda", dtype=torch.float64)
    u = torch.rand((200_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    r.deposit(torch.cat([torch.remainder(p, L), u]))
    return r


def _rel(a, b):
    return float((a - b).double().norm() / b.double().norm())


def _both(r, fn):
    from paper_1504_02591_gb300 import binding as B
    out = []
    for generic in (1, 0):
        r.set_option(B.OPT_KSPACE_GENERIC, generic)
        out.append(fn())
    return out


@pytest.mark.parametrize("n,los,tile,planes", [(256, 0, 0, 0), (256, 1, 1, 32), (384, 0, 1, 0), (384, 1, 0, 16), (512, 1, 1, 0),
                                               (512, 0, 0, 64), (1024, 0, 0, 0), (1024, 1, 1, 0)])
def test_fused_iteration_matches_generic(lib, n, los, tile, planes):
    from paper_1504_02591_gb300 import binding as B
    r = _box(n, los)
    r.set_option(B.OPT_LINE_TILE, tile)
    r.set_option(B.OPT_PLANE_BATCH, planes)
    r.smooth()

    def run():
        n_it, rel, _ = r.iterate(B.START_FFTA, 0.0, 3)
        return r.get_psi(), r.trace()

    (psi_g, tr_g), (psi_f, tr_f) = _both(r, run)
    assert _rel(psi_f, psi_g) < TOL
    assert max(abs(a / b - 1) for a, b in zip(tr_f, tr_g)) < 1e-3
    # the host-driven loop ends in its own final pass
    r.set_option(B.OPT_GRAPH, 0)
    r.iterate(B.START_FFTA, 0.0, 3)
    assert torch.equal(r.get_psi(), psi_f)
    r.close()


@pytest.mark.parametrize("n,los,level", [(256, 0, 2), (384, 0, 1), (384, 1, 2), (1024, 0, 2)])
def test_fused_warm_start_matches_generic(lib, n, los, level):
    from paper_1504_02591_gb300 import binding as B
    r = _box(n, los)
    rho = r.get_field(B.FIELD_RHO_G)
    assert float(rho.sum()) == pytest.approx(456_000, rel=1e-4)

    def run():
        r.smooth()
        feat = r.start_features(B.START_FFTA, level)
        u0 = feat[..., 4] * 1.1 + 0.2 * feat[..., 0]
        r.iterate_from(u0.contiguous(), 0.0, 2, level)
        warm, u = r.get_psi(), r.get_radial(0)
        r.iterate_from(u, 0.0, 2, 0)
        return feat, warm, r.get_psi()

    out = []
    for generic in (1, 0):
        r.close()
        r = _box(n, los)
        r.set_option(B.OPT_KSPACE_GENERIC, generic)
        out.append(run())
    for g, f in zip(*out):
        assert _rel(f, g) < TOL
    r.close()
