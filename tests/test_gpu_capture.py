"""recon_start_features inside a caller's CUDA graph: it is captured, and its replay gives what the call gives."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 256])   # generic kernels, streamed ones
def test_start_features_in_a_captured_stream(lib, n):
    from paper_1504_02591_gb300 import binding as B
    L = 6.0 * n
    g = torch.Generator(device="cuda").manual_seed(n)
    gal = torch.rand((50_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        r = B.Recon(n, L, 1.6, 0.7, 15.0, (-0.3 * L, 0.5 * L, 0.4 * L), periodic=True, uniform=True)
        r.deposit(gal)
        r.smooth()
        want = r.start_features(B.START_FFTA, 1)
        r.deposit(gal)
        r.smooth()
        s.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            got = r.start_features(B.START_FFTA, 1)
        graph.replay()
        s.synchronize()
    # only the deposit's order of float32 sums differs
    assert float((got - want).norm() / want.norm()) < 1e-5
    r.close()
