"""The brick-sorted shift, on request (RECON_PATH_SORTED sorts whatever the mesh and the catalogue; the automatic
path only where it pays): images of the box, float32 positions, boxes that do not wrap, both lines of sight,
several chunks and the parts of a host result.  Reference: the direct gather of the same positions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solved(n, L, los="radial", periodic=True):
    from paper_1504_02591_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(n)
    gal = torch.rand((60_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    obs, mode = ((-0.5 * L, 0.4 * L, 0.7 * L), B.LOS_RADIAL) if los == "radial" else ((0.6, 0.0, 0.8), B.LOS_FIXED)
    r = B.Recon(n, L, 1.6, 0.7, 2.5 * L / n, obs, los_mode=mode, periodic=periodic, uniform=True)
    r.run(gal, None, B.START_FFTA, 0.0, 1)
    return r


def _tolerance(r):
    """Three axes, one unit of the 21-bit fraction each, times the largest step of Psi between nodes, in the
    three components that the redshift-space term adds up (1 + 0.7 sqrt 3 < 2.3); and in each path ten roundings
    of half a unit in the interpolation and 0.7 times ten units in that term, 24 units of 2^-24 together."""
    psi = r.get_psi()
    step = max(float((psi - torch.roll(psi, 1, a)).abs().max()) for a in (1, 2, 3))
    return 2.3 * 3 * 2.0 ** -21 * step + 24 * 2.0 ** -24 * float(psi.abs().max())


def _sorts(r):
    return r.timing()["sort"][0]


@pytest.mark.parametrize("n,count,dtype,los,periodic,host", [
    (32, 1, np.float64, "radial", True, False),
    (48, 1031, np.float32, "radial", True, False),
    (64, 200_003, np.float64, "fixed", False, True),
    (48, (1 << 22) + 77, np.float32, "radial", False, False),      # two chunks of the sort
    (128, (1 << 21) + 5, np.float64, "radial", True, True),        # two staged chunks
    (256, 300_001, np.float32, "fixed", True, False),
    (512, 100_001, np.float64, "radial", True, False),
])
def test_sorted_shift_equals_direct(lib, n, count, dtype, los, periodic, host):
    from paper_1504_02591_gb300 import binding as B
    L = 6.0 * n
    r = _solved(n, L, los, periodic)
    tol = _tolerance(r)
    rng = np.random.default_rng(count)
    pos = rng.uniform(0.0, L, (count, 3))
    k = min(count, 600)
    pos[:k] += L * rng.integers(-2, 3, (k, 3))                     # images of the box
    pos[k // 2:k // 2 + 8, 0] = [0.0, L, np.nextafter(L, 0), -0.0, L / n, 8 * L / n, L - 8 * L / n, -L][:max(0, min(8, count - k // 2))]
    pos = np.ascontiguousarray(pos.astype(dtype))
    p = pos if host else torch.from_numpy(pos).cuda()
    for galaxy in (True, False):
        out = {}
        for path in (B.PATH_DIRECT, B.PATH_SORTED):
            r.set_option(B.OPT_SHIFT_PATH, path)
            s0 = _sorts(r)
            d, y = r.shift(p, galaxy, want_pos=True)
            chunks = -(-count // (min(1 << 21, 1 << 22 if n < 256 else 1 << 25) if host else (1 << 22 if n < 256 else 1 << 25)))
            assert _sorts(r) - s0 == (chunks if path == B.PATH_SORTED else 0)
            d, y = np.asarray(d if host else d.cpu()), np.asarray(y if host else y.cpu())
            out[path] = d
            want = pos.astype(np.float64) + d
            if periodic:
                want = want - np.floor(want / L) * L
                want = np.where(want >= L, want - L, want)
            assert np.array_equal(y, want)
        assert np.abs(out[B.PATH_DIRECT] - out[B.PATH_SORTED]).max() <= tol
    r.close()


def test_automatic_path_sorts_by_size(lib):
    from paper_1504_02591_gb300 import binding as B
    n = 384
    r = _solved(n, 6.0 * n)
    g = torch.Generator(device="cuda").manual_seed(2)
    pos = torch.rand((n ** 3 // 32, 3), generator=g, device="cuda", dtype=torch.float64) * 6.0 * n
    for count, sorts in ((n ** 3 // 32 - 1, 0), (n ** 3 // 32, 1)):
        s0 = _sorts(r)
        r.shift(pos[:count], True)
        assert _sorts(r) - s0 == sorts
    for bad in (-1, 3):
        with pytest.raises(B.ReconError) as e:
            r.set_option(B.OPT_SHIFT_PATH, bad)
        assert e.value.status == B.ERR_INVALID_ARG
    r.close()


def test_retained_order_to_host_in_parts(lib):
    """A retained order's shifts leave for host memory through a staging buffer of 2 x 2^21 x 64 bytes: 23e6
    tracers take two parts, which hold the same values as the device result."""
    from paper_1504_02591_gb300 import binding as B
    n, count = 256, 23_000_003
    assert count > 2 * (1 << 21) * 64 // 12
    L = 6.0 * n
    g = torch.Generator(device="cuda").manual_seed(5)
    pos = torch.rand((count, 3), generator=g, device="cuda", dtype=torch.float32) * L
    host = pos.cpu().pin_memory()
    r = _solved(n, L)
    r.set_option(B.OPT_DEPOSIT_PATH, B.PATH_SORTED)
    r.set_option(B.OPT_REUSE_SORT, 1)
    r.deposit(host)
    r.smooth()
    r.iterate(B.START_FFTA, 0.0, 1)
    s0 = _sorts(r)
    a = torch.as_tensor(r.shift(host, True))
    assert _sorts(r) == s0
    r.set_option(B.OPT_REUSE_SORT, 0)
    r.set_option(B.OPT_SHIFT_PATH, B.PATH_SORTED)
    b = r.shift(pos, True)
    assert torch.equal(a, b.cpu())
    r.close()


def test_automatic_path_decides_by_chunk(lib):
    """Chunks are sorted one by one, so a chunk's own size decides: staged chunks of 2^21 tracers on a 512 mesh
    (N^3 / 32 is twice that) and the short last chunk of a device catalogue are gathered directly."""
    from paper_1504_02591_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(7)
    for n, count, device_sorts, host_sorts in ((512, 512 ** 3 // 32 + 1, 1, 0), (384, (1 << 25) + 1001, 1, None)):
        r = _solved(n, 6.0 * n)
        tol = _tolerance(r)
        pos = torch.rand((count, 3), generator=g, device="cuda", dtype=torch.float32) * 6.0 * n
        s0 = _sorts(r)
        a = r.shift(pos, True)
        assert _sorts(r) - s0 == device_sorts
        if host_sorts is not None:
            s0 = _sorts(r)
            b = torch.as_tensor(r.shift(pos.cpu().numpy(), True))
            assert _sorts(r) - s0 == host_sorts
            assert float((a.cpu() - b).abs().max()) <= tol
        else:
            r.set_option(B.OPT_SHIFT_PATH, B.PATH_DIRECT)
            assert float((a - r.shift(pos, True)).abs().max()) <= tol
        r.close()
