"""The finite-difference solve works in pairs of float32; the units of length and of the bias, and an observer
at any distance, must not take them out of float32's range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve(n, L, b, observer, los, scale=1.0):
    from paper_1504_02591_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(12)
    gal = torch.rand((40_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    gal[:20_000] = gal[:20_000] * 0.25 + 0.3 * L
    r = B.Recon(n, L * scale, b, 0.37 * b, 2.2 * L / n * scale, tuple(v * scale for v in observer), los_mode=los,
                periodic=True, uniform=True)
    r.deposit(gal * scale)
    r.smooth()
    psi, it, res, st = r.fd_solve(1e-5, 200)
    r.close()
    assert st == B.OK and np.isfinite(res) and it > 2
    return psi.double() / scale


def _rel(a, b):
    return float((a - b).norm() / b.norm())


# The deposits add in any order, so two solves of the same catalogue differ by the solver's tolerance at most:
# |A phi - b| <= 1e-5 |b| each, plus float32's floor of the residual near 1e-5.
@pytest.mark.parametrize("n,power,los", [(32, 56, "radial"), (32, -58, "radial"), (48, 55, "fixed"), (32, -58, "fixed")])
def test_units_of_length(lib, n, power, los):
    """L, R, the observer and the positions times a power of two: the same Psi times it.  2^56: the squared
    offsets pass float32's range; 2^-58: their low halves and the operator's are subnormal."""
    from paper_1504_02591_gb300 import binding as B
    L = 6.0 * n
    obs, mode = ((-0.7 * L, 0.4 * L, 0.6 * L), B.LOS_RADIAL) if los == "radial" else ((0.6, 0.0, 0.8), B.LOS_FIXED)
    want = _solve(n, L, 1.7, obs, mode)
    scale = 2.0 ** power
    if los == "fixed":
        obs = tuple(v / scale for v in obs)          # a direction: not a length
    assert _rel(_solve(n, L, 1.7, obs, mode, scale), want) < 1e-4


@pytest.mark.parametrize("distance", [1e12, 1e21, 1e30])
def test_distant_observer_is_a_fixed_line_of_sight(lib, distance):
    from paper_1504_02591_gb300 import binding as B
    want = _solve(32, 200.0, 1.7, (1.0, 0.0, 0.0), B.LOS_FIXED)
    assert _rel(_solve(32, 200.0, 1.7, (-distance, 100.0, 100.0), B.LOS_RADIAL), want) < 1e-4


def test_observer_on_a_node(lib):
    """The line-of-sight term is zero there."""
    from paper_1504_02591_gb300 import binding as B
    assert bool(torch.isfinite(_solve(32, 192.0, 1.7, (96.0, 96.0, 96.0), B.LOS_RADIAL)).all())


def test_unit_of_the_bias(lib):
    """delta / b far below the range in which squares keep their digits: Psi is delta's, over b (f / b fixed)."""
    from paper_1504_02591_gb300 import binding as B
    obs = (-140.0, 80.0, 110.0)
    want = _solve(32, 200.0, 1.0, obs, B.LOS_RADIAL)
    assert _rel(_solve(32, 200.0, 2.0 ** 60, obs, B.LOS_RADIAL) * 2.0 ** 60, want) < 1e-4
