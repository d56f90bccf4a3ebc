"""Radial shells and FKP weights where the float32 offsets are hard: observers at the origin, on the particles'
planes and far away, coordinates of exactly zero, remainders of the four-particle batches."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("count,obs", [(1, (0.0, 0.0, 0.0)), (1023, (0.0, 50.0, 50.0)), (300_001, (-1e6, 3e5, 2e6)),
                                       (300_001, (-1e12, 0.0, 0.0))])
def test_shells_match_float64(dtype, count, obs):
    """A weight is the table's value of the particle's float64 shell, exactly, unless its distance is at an edge
    to float64 rounding: 1e-12 of the shells' coordinate, taken from (r / dr) 2^-50."""
    from paper_1504_02591_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(count)
    pos = (torch.rand((count, 3), generator=g, device="cuda", dtype=torch.float64) * 100.0).to(dtype)
    pos[::7, 1] = 0.0
    x = pos.double().cpu().numpy() - np.array(obs)
    r = np.sqrt((x * x).sum(1))
    nbins, rmin = 37, float(r.min()) * 0.999
    rmax = max(float(r.max()) * 0.9995, rmin + 1e-3)
    table = np.linspace(1e-4, 3e-3, nbins)
    h = B.Recon(32, 100.0, 1.8, 0.7, 15.0, obs, 0, True, 0.01, False, True)
    w = h.fkp_weights(pos, table, rmin, rmax, 1e4).cpu().numpy()
    h.close()
    f = (r - rmin) * (nbins / (rmax - rmin))
    b = np.floor(f)
    inside = (b >= 0) & (b < nbins)
    want = (1.0 / (1.0 + np.where(inside, table[np.clip(b, 0, nbins - 1).astype(int)], 0.0) * 1e4)).astype(np.float32)
    edge = np.abs(f - np.rint(f)) <= np.maximum(1e-12 * np.abs(f), r * (nbins / (rmax - rmin)) * 2.0 ** -50)
    assert (np.abs(w / want - 1) <= 1e-7)[~edge].all()
