"""Particle arithmetic that leaves the plain float64 path: the fixed-point coordinates from one rounded-down
multiply-add, the wrap of shifted positions without a division, and shells found in float32 away from
their edges; and the routes a shift can take.  Each is compared with the float64 expression it stands for, at the places where it could
go wrong: box edges, images of the box (near and hundreds of boxes away, past the 2^51 range of the
multiply-add), shell edges, the observer itself and remainders of the launch sizes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _positions(L, n, count, dtype, seed):
    rng = np.random.default_rng(seed)
    p = rng.uniform(0.0, L, (count, 3))
    edge = np.array([0.0, L * (1 - 2.0 ** -50), L / n, L * (n - 1) / n, L * 0.5, L / (2 * n), np.nextafter(L, 0)])
    k = len(edge)
    p[:k, 0], p[k:2 * k, 1], p[2 * k:3 * k, 2] = edge, edge, edge
    p[3 * k:3 * k + 50] += L * rng.integers(-3, 4, (50, 3))
    p[3 * k + 50:3 * k + 60] += L * 3.0e6                       # past the multiply-add's range at any mesh
    p[3 * k + 60:3 * k + 70] -= L * 700.0
    return p.astype(dtype)


@pytest.mark.parametrize("n,count,dtype", [(32, 1000, np.float64), (96, 257, np.float32), (256, 20011, np.float64)])
@pytest.mark.parametrize("path", [0, 1])
def test_deposit_of_edges_and_images(lib, n, count, dtype, path):
    """CIC weights are continuous across cells, so rounding in the last bit of a coordinate moves no mass
    beyond 2^-20 of a cell (21 fraction bits on the sorted path); images far away carry the coordinate's own
    float64 spacing."""
    from paper_1504_02591_gb300 import binding as B
    L = 700.0
    pos = _positions(L, n, count, dtype, 3)
    r = B.Recon(n, L, 1.5, 0.7, 10.0, (-500.0, 300.0, 200.0), uniform=True)
    r.set_option(B.OPT_DEPOSIT_PATH, path)
    w = np.linspace(0.5, 1.5, count).astype(np.float32)
    for weights in (None, w):
        r.deposit(torch.from_numpy(pos).cuda(), None if weights is None else torch.from_numpy(weights).cuda())
        rho = r.get_field(B.FIELD_RHO_G).cpu().numpy().astype(np.float64)
        ww = np.ones(count) if weights is None else weights.astype(np.float64)
        assert r.scalars()["sum_wg"] == pytest.approx(ww.sum(), rel=1e-14)
        u = pos.astype(np.float64) * (n / L)
        i0 = np.floor(u)
        t = u - i0
        ref = np.zeros(n ** 3)
        for d in range(8):
            o = [(d >> 2) & 1, (d >> 1) & 1, d & 1]
            c = np.ones(count)
            idx = np.zeros(count, dtype=np.int64)
            for a in range(3):
                c = c * (t[:, a] if o[a] else 1 - t[:, a])
                idx = idx * n + ((i0[:, a].astype(np.int64) + o[a]) % n)
            np.add.at(ref, idx, ww * c)
        # per node: the fraction's 2^-21 (floor) on each of its particles, and float32 sums
        tol = 3 * 2.0 ** -21 * 1.5 * 8 + 1e-6 * np.abs(ref).max()
        assert np.abs(rho.ravel() - ref).max() < tol + 10 * 1.5 * 3e6 * n * 2.0 ** -52
    r.close()


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("dtype,path", [(np.float64, 0), (np.float32, 1), (np.float64, 1)])
def test_shifted_positions_wrap(lib, periodic, dtype, path):
    """pos_out is exactly y - floor(y / L) L (stepped back from L) of y = position + shift in float64."""
    from paper_1504_02591_gb300 import binding as B
    n, L = 48, 600.0
    g = torch.Generator(device="cuda").manual_seed(4)
    gal = torch.rand((30_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    r = B.Recon(n, L, 1.2, 0.8, 8.0, (-700.0, 300.0, 280.0), periodic=bool(periodic), uniform=True)
    r.run(gal, None, B.START_FFTA, 0.0, 2)
    r.set_option(B.OPT_SHIFT_PATH, path)
    pos = torch.from_numpy(_positions(L, n, 1031, dtype, 9)).cuda()
    d, out = r.shift(pos, True, want_pos=True)
    y = pos.double() + d.double()
    if periodic:
        y = y - torch.floor(y / L) * L
        y = torch.where(y >= L, y - L, y)
    assert torch.equal(out, y)
    r.close()


@pytest.mark.parametrize("nbins,rmin,rmax", [(1, 100.0, 900.0), (50, 150.0, 640.0), (4096, 0.0, 800.0)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_shells_match_float64(lib, nbins, rmin, rmax, dtype):
    from paper_1504_02591_gb300 import binding as B
    L, P0 = 1000.0, 12345.0
    obs = np.array([0.0, 500.0, 480.0])
    rng = np.random.default_rng(nbins)
    pos = rng.uniform(0.0, L, (40_003, 3))
    # on shell edges, up to float64 rounding, along random directions; and the observer itself
    v = rng.standard_normal((6000, 3))
    v /= np.linalg.norm(v, axis=1)[:, None]
    pos[:6000] = obs + v * (rmin + (rmax - rmin) / nbins * rng.integers(0, nbins + 1, 6000))[:, None]
    pos[6000] = obs
    pos = pos.astype(dtype)
    r = B.Recon(32, L, 1.5, 0.7, 10.0, tuple(obs), uniform=True)
    t = torch.from_numpy(pos).cuda()
    d = t.double() - torch.from_numpy(obs).cuda()
    # the edge cases are decided by the last bit: the same fused float64 expression on the GPU
    rr = torch.sqrt(torch.addcmul(torch.addcmul(d[:, 2] * d[:, 2], d[:, 1], d[:, 1]), d[:, 0], d[:, 0]))
    b = torch.floor((rr - rmin) * (nbins / (rmax - rmin))).cpu().numpy()
    inside = (b >= 0) & (b < nbins)
    nbar = r.radial_nbar(t, nbins, rmin, rmax, 1.7)
    e = rmin + (rmax - rmin) / nbins * np.arange(nbins + 1)
    counts = nbar * (1.7 * (e[1:] ** 3 - e[:-1] ** 3) / 3)
    want = np.bincount(b[inside].astype(int), minlength=nbins)
    # a particle on an edge to the last bit may fall either way (the sum's order): at most those
    on_edge = np.abs((rr.cpu().numpy() - rmin) * (nbins / (rmax - rmin)) - np.rint((rr.cpu().numpy() - rmin) * (nbins / (rmax - rmin)))) < 1e-9 * nbins
    assert np.abs(np.rint(counts) - want).sum() <= 2 * on_edge.sum()
    table = np.append(rng.uniform(1e-5, 1e-2, nbins), 0.0)
    w = r.fkp_weights(t, table[:nbins], rmin, rmax, P0).cpu().numpy()
    ref = (1.0 / (1.0 + table[np.where(inside, b, nbins).astype(int)] * P0)).astype(np.float32)
    ok = (w == ref) | (np.abs(w / ref - 1) < 1e-7)
    assert ok[~on_edge].all()
    r.close()


@pytest.mark.parametrize("n,count", [(64, 200_000), (96, 250_001), (256, 2_097_152), (384, 1_769_472)])
def test_shift_routes_agree(lib, n, count):
    """At the sizes where a shift changes its route (direct, packed nodes, sorted) it gives the values of the
    route below: packed nodes the same bits (the same products in the same order), the sorted gather up to
    its 21-bit fractions."""
    from paper_1504_02591_gb300 import binding as B
    L = 6.0 * n
    g = torch.Generator(device="cuda").manual_seed(n)
    gal = torch.rand((60_000, 3), generator=g, device="cuda", dtype=torch.float64) * L
    r = B.Recon(n, L, 1.6, 0.7, 12.0, (-0.5 * L, 0.4 * L, 0.7 * L), periodic=True, uniform=True)
    r.run(gal, None, B.START_FFTA, 0.0, 1)
    pos = torch.rand((count, 3), generator=g, device="cuda", dtype=torch.float64) * L
    for galaxy in (True, False):
        d, y = r.shift(pos, galaxy, want_pos=True)
        few, yf = r.shift(pos[:count - 1].contiguous()[:1000], galaxy, want_pos=True)
        if n < 384:
            assert torch.equal(d[:1000], few) and torch.equal(y[:1000], yf)
        else:
            psi = r.get_psi()
            step = max(float((psi - torch.roll(psi, 1, a)).abs().max()) for a in (1, 2, 3))
            # three axes, half a unit of the fraction on average and one at most; 1.7: the redshift-space factor
            tol = 3 * 2.0 ** -21 * step * 1.7 + 4e-7 * float(psi.abs().max()) * 1.7
            assert float((d[:1000] - few).abs().max()) < tol
            assert float((y[:1000] - yf).abs().max()) < tol + 1e-12
    r.close()


def test_retained_order_shift_to_host_and_device(lib):
    """The retained brick order serves device and host outputs, and survives a shift of another catalogue."""
    from paper_1504_02591_gb300 import binding as B
    n, L = 128, 900.0
    g = torch.Generator(device="cuda").manual_seed(8)
    pos = torch.rand((150_003, 3), generator=g, device="cuda", dtype=torch.float64) * L
    host = pos.cpu().pin_memory()
    r = B.Recon(n, L, 1.6, 0.7, 12.0, (-400.0, 300.0, 500.0), periodic=True, uniform=True)
    r.run(pos, None, B.START_FFTA, 0.0, 1)
    ref = r.shift(pos, True)
    r.set_option(B.OPT_DEPOSIT_PATH, B.PATH_SORTED)
    r.set_option(B.OPT_REUSE_SORT, 1)
    for src in (pos, host):
        r.deposit(src)
        r.smooth()
        r.iterate(B.START_FFTA, 0.0, 1)
        other = r.shift(pos[:777].contiguous(), True)
        a, b = r.shift(src, True), r.shift(src, True)
        a, b = (torch.as_tensor(v).cuda() for v in (a, b))
        assert torch.equal(a, b)
        assert float((a - ref).abs().max()) < 1e-4 * float(ref.abs().max())
        assert float((other - ref[:777]).abs().max()) < 1e-4 * float(ref.abs().max())
    r.close()
