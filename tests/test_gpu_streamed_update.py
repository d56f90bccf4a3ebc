"""The source update with its inputs streamed into shared memory (RECON_OPT_KITER_TMA 1, the default of the
meshes of the register-fused family) against the update with direct loads, on every mesh of the family."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [256, 384, 1024])
def test_streamed_update_matches_direct_loads(n):
    """Element for element the same arithmetic: Psi is bitwise equal (the 1024 mesh has narrower tiles and
    four boxes a line, 384 boxes of 192 rows).  Both group float32 squares of up to 24 values per thread
    before wider sums, so the norms agree to 24 roundings, 24 * 6e-8 = 1.5e-6."""
    from paper_1504_02591_gb300 import binding as B
    side = 6.84 * n
    r = B.Recon(n, side, 1.8, 0.7, 15.0, (-0.5 * side, 0.4 * side, 0.6 * side), 0, True, 0.01, False, True)
    g = torch.Generator(device="cuda").manual_seed(n)
    pos = torch.rand((300_000, 3), generator=g, device="cuda", dtype=torch.float64) * side
    r.deposit(pos)
    r.smooth()
    out = []
    for tma in (1, 0):
        r.set_option(B.OPT_KITER_TMA, tma)
        r.iterate(B.START_FFTA, 0.0, 3)
        out.append((r.get_psi().cpu().numpy(), np.array(r.trace())))
    r.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.allclose(out[0][1], out[1][1], rtol=1.5e-6, atol=0)
