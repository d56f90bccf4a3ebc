"""The batch autotuner leaves open what its first mock cannot decide: a small first catalogue does not pin the
direct shift for the larger ones of its mesh, and schedules that run the same kernels are not told apart by
timing noise (one tile width in the streamed x passes, the generic kernels alone in the alternative radix order)."""
import pytest

from paper_1504_02591_gb300 import mocks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [96, 128, 256, 384])
def test_small_first_catalogue_pins_nothing(lib, n):
    from paper_1504_02591_gb300 import binding as B
    m = mocks.batch_mock_device(n, 5_000, 10, 1.8, 0.7, False, n)
    status, res = B.batch_run([m], start=B.START_FFTA, tol=0.0, max_iter=2)
    assert status == B.OK and res[0]["n_iter"] == 2
    plan = B.batch_plan(n)
    assert plan["shift_path"] == B.PATH_AUTO
    if n >= 256 and plan["fft_radix"] == 0:
        assert plan["line_tile"] == 0
