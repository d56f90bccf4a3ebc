"""The bounded waits of the streamed kernels (RECON_OPT_DROP_COPY leaves out one tile's copy, so a wait runs
out; the copy of a later tile is then on its way): the call returns RECON_ERR_TIMEOUT, also where no norm
follows the pass, and the handle works again from the next deposit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("drop,graph", [(1, 1), (1, 0), (2, 1)])
def test_a_wait_that_runs_out_is_reported(lib, drop, graph):
    from paper_1504_02591_gb300 import binding as B
    n, L = 256, 1500.0
    g = torch.Generator(device="cuda").manual_seed(3)
    gal = torch.rand((100_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    r = B.Recon(n, L, 1.6, 0.7, 15.0, (-400.0, 700.0, 800.0), periodic=True, uniform=True)
    r.set_option(B.OPT_GRAPH, graph)

    def start():
        r.deposit(gal)
        r.smooth()

    start()
    r.iterate(B.START_FFTA, 0.0, 2)
    want = r.get_psi()
    r.set_option(B.OPT_DROP_COPY, drop)
    start()
    if drop == 1 and graph:
        with pytest.raises(B.ReconError) as e:   # its inverse x pass is followed by no norm
            r.start_features(B.START_FFTA, 1)
        assert e.value.status == B.ERR_TIMEOUT
    with pytest.raises(B.ReconError) as e:
        r.iterate(B.START_FFTA, 0.0, 2)
    assert e.value.status == B.ERR_TIMEOUT
    with pytest.raises(B.ReconError) as e:
        r.shift(gal, True)
    assert e.value.status == B.ERR_STATE
    r.set_option(B.OPT_DROP_COPY, 0)
    start()
    n_it, rel, st = r.iterate(B.START_FFTA, 0.0, 2)
    assert n_it == 2 and np.isfinite(rel)
    # only the deposit's order of float32 sums differs
    assert float((r.get_psi() - want).norm() / want.norm()) < 1e-5
    r.close()
