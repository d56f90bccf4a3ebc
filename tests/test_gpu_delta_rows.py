"""The z factor of the smoothing with delta and its r2c: the register-fused rows against the generic pass on
every mesh of the family, from few taps to the most that the fused rows take."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,uniform,lognormal", [(256, 2.2, True, False), (256, 4.8, False, False), (384, 0.4, False, True),
                                                   (384, 4.8, True, True), (512, 4.2, False, True), (1024, 4.1, True, False),
                                                   (1024, 2.2, False, False)])
def test_delta_rows_match_generic(n, R, uniform, lognormal):
    """Points at half-integer node offsets deposit multiples of 1/8, so the density is the same to the bit both
    times, and both passes add the taps in the same order: q = 1 + delta differs by the contraction of its
    last product and sum at most, 2^-23 (1 + |delta|); the logarithm adds an ulp of its own, 2^-23 (1 + |d|).
    4e-7 (1 + |delta|) bounds both.  delta(k) then differs by the rounding of two float32 transforms (3.3e-7
    each in the L2 norm at most, as 3 log2 N levels of 6e-8 in quadrature) and by that of delta."""
    from paper_1504_02591_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(n)
    pos = [torch.randint(0, 2 * n, (c, 3), generator=g, device="cuda").double() / 2 for c in (300_000, 2_000_000)]
    # the randoms leave a slab empty, so that some nodes are outside the mask
    pos[1][:, 2] *= 0.75
    pos[1] = torch.floor(2 * pos[1]) / 2
    r = B.Recon(n, float(n), 1.8, 0.7, R, (-0.5 * n, 0.4 * n, 0.6 * n), 0, uniform, 0.01, lognormal, uniform)
    out = []
    for generic in (1, 0):
        r.set_option(B.OPT_KSPACE_GENERIC, generic)
        r.deposit(pos[0], None, None if uniform else pos[1], None)
        r.smooth()
        d = r.get_field(B.FIELD_DELTA)
        r.iterate(B.START_FFTA, 0.0, 1)
        out.append((d, r.get_field(B.FIELD_DELTA_K)))
    r.close()
    (dg, kg), (df, kf) = out
    assert bool(((df - dg).abs() <= 4e-7 * (1 + dg.abs())).all())
    assert float(torch.view_as_real(kf - kg).double().norm() / torch.view_as_real(kg).double().norm()) < 1.5e-6
