"""The convergence norms: the sum of an update's partials by one block and by several, with the decision in the
same kernel (graph loop) and without (host loop)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tma", [(32, 1), (64, 1), (256, 1), (256, 0), (384, 0)])
def test_graph_and_host_loops_see_the_same_norms(n, tma):
    """Both loops sum the same partials in the same order, so the traces are equal to the bit; rel of the last
    update is also that of the k-space sums of the sources, which the next Psi differs by: |dPsi| / |Psi| from
    two runs that stop one update apart.  Psi is float32, so its difference of relative size rel carries up to
    2^-23 / rel of rounding; the runs keep rel above 1e-3, so 1e-3 bounds it."""
    from paper_1504_02591_gb300 import binding as B
    side = 6.84 * n
    r = B.Recon(n, side, 1.8, 0.7, 15.0, (-0.5 * side, 0.4 * side, 0.6 * side), 0, True, 0.01, False, True)
    r.set_option(B.OPT_KITER_TMA, tma)
    g = torch.Generator(device="cuda").manual_seed(n)
    r.deposit(torch.rand((100_000, 3), generator=g, device="cuda", dtype=torch.float64) * side)
    r.smooth()
    out = []
    for graph in (1, 0):
        r.set_option(B.OPT_GRAPH, graph)
        r.iterate(B.START_FFTA, 0.0, 3)
        out.append((np.array(r.trace()), r.get_psi().double()))
    assert np.array_equal(out[0][0], out[1][0])
    r.iterate(B.START_FFTA, 0.0, 2)
    last = r.get_psi().double()
    r.close()
    rel = float(torch.linalg.vector_norm(out[0][1] - last) / torch.linalg.vector_norm(out[0][1]))
    assert out[0][0][-1] > 1e-3
    assert abs(rel / out[0][0][-1] - 1) < 1e-3
