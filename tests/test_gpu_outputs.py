"""The output kernels at the sizes where their fast forms can go wrong: the
power spectrum's mixed-radix rows, the histogram's and the momentum spectrum's
FP32 bins with values on bin edges, and the energy and stability sums, against
numpy on the run's own field and particles."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_14282_gb300 import build
    build.build()
    from paper_2507_14282_gb300 import fs as m
    return m


# rows of one radix each, of all of them, with a large prime factor (167, 61),
# with two (43 x 47), left to the direct DFT (2 x 3541), the longest in shared
# memory and one beyond it
ROWS = [(2, 3), (4, 2), (6, 1), (49, 2), (60, 5), (125, 2), (210, 3), (512, 2), (1002, 4), (2021, 2),
        (3000, 2), (7082, 1), (122, 200), (14400, 1), (14402, 1)]


@pytest.mark.parametrize("nx,ny", ROWS, ids=lambda v: str(v))
@pytest.mark.parametrize("prec", [0, 1])
def test_spectrum_rows(fs, nx, ny, prec):
    rng = np.random.default_rng(nx + ny)
    B = rng.normal(size=(ny, nx, 3))
    if prec:
        B = B.astype(np.float32).astype(np.float64)
    # a short row takes any tile that divides it; long prime rows need one given
    sim = fs.FauxShock(dim=2, nx=nx, ny=ny, ppc=1, precision=prec, init_plasma=0)
    sim.load_fields(B)
    got, want = sim.grid(fs.FS_SPECTRUM_BPERP), O.bperp_spectrum(B)
    # FP64 sums of up to 14402 terms: rounding of order 1e-16 sqrt(n) of the row's power
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-12 * want.max())
    np.testing.assert_array_equal(sim.grid(fs.FS_PROFILE_DB2).shape, (nx,))
    sim.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dim,nx,ny,hist,spec", [
    (1, 96, 1, (7, 33), 17), (1, 1000, 1, (1000, 3), 2000), (2, 60, 35, (64, 64), 64),
    (2, 48, 18, (1, 20000), 9000), (2, 24, 80, (300, 128), 1)])
def test_counts_equal_numpy(fs, prec, dim, nx, ny, hist, spec):
    """Whole counts: the written FP64 expressions on every particle."""
    kw = dict(dim=dim, nx=nx, ny=ny, ppc=6, precision=prec, capacity_factor=60.0,
              hist_nx=hist[0], hist_np=hist[1], hist_pmin=-30.0, hist_pmax=50.0, spec_np=spec,
              spec_pmin=0.5, spec_pmax=400.0)
    sim = fs.FauxShock(**kw)
    rng = np.random.default_rng(spec)
    # values on and beside the edges of both binnings, cosmic rays, and a few far outside
    pe = -30.0 + 80.0 / hist[1] * rng.integers(-2, hist[1] + 3, 500)
    ue = 0.5 * 800.0 ** (rng.integers(0, spec + 1, 500) / spec)
    vx = np.concatenate([pe, np.nextafter(pe, -1e9), np.nextafter(pe, 1e9), 0 * ue, [1e7, -1e7, 0]])
    vy = np.concatenate([rng.normal(size=1500), ue, [0, 1e-9, 0]])
    n = len(vx)
    fx = np.where(rng.random(n) < 0.3, rng.integers(0, 4, n) / 4.0, rng.random(n))
    sim.inject(rng.integers(0, nx, n), rng.integers(0, ny, n), fx, rng.random(n), vx, vy,
               np.zeros(n), ids=((nx * ny * 6 + np.arange(n)) | np.where(
                   rng.random(n) < 0.5, fs.ID_CR, 0)).astype(np.uint32))
    p = sim.particles()
    cr = (p["id"] & fs.ID_CR) != 0
    bx = np.clip(np.floor((p["ci"] + p["fx"]) * (hist[0] / nx)).astype(int), 0, hist[0] - 1)
    bp = np.floor((p["vx"] - -30.0) * (hist[1] / 80.0))
    ok = (bp >= 0) & (bp < hist[1])
    for only in (False, True):
        m = ok & (cr | (not only))
        want = np.zeros(hist, np.int64)
        np.add.at(want, (bx[m], bp[m].astype(int)), 1)
        np.testing.assert_array_equal(sim.histogram(cr_only=only), want)
    # |u| as the spectrum forms it, to the last bit but for its fused sums: a value
    # within 4 ulp of an edge may fall on either side
    u = np.sqrt(p["vx"] ** 2 + p["vy"] ** 2 + p["vz"] ** 2)
    edges = 0.5 * np.exp(np.arange(spec + 1) / spec * np.log(800.0))
    lo = np.searchsorted(edges, u * (1 - 1e-15), side="right") - 1
    hi = np.searchsorted(edges, u * (1 + 1e-15), side="right") - 1
    for only in (False, True):
        got = sim.spectrum_p(cr_only=only)
        m = cr if only else np.ones_like(cr)
        sure = m & (lo == hi) & (lo >= 0) & (lo < spec)
        want = np.bincount(lo[sure], minlength=spec)[:spec]
        loose = np.zeros(spec + 2, np.int64)
        for k in (lo, hi):
            np.add.at(loose, np.clip(k[m & (lo != hi)], -1, spec) + 1, 1)
        assert ((got >= want) & (got <= want + loose[1:-1])).all()
    w = np.where(cr, 0.01, 1.0) / 6 * 0.5 ** dim
    d = sim.diag()
    v2 = (w * (p["vx"] ** 2 + p["vy"] ** 2 + p["vz"] ** 2)).sum() / 2
    assert abs(d["kinetic"] - v2) <= 1e-12 * v2
    for k in ("vx", "vy", "vz"):
        assert abs(d["p" + k[1]] - (w * p[k]).sum()) <= 1e-12 * (w * np.abs(p[k])).sum()
    sim.close()


@pytest.mark.parametrize("dim,nx,ny,prec", [(1, 4000, 1, 1), (1, 640, 1, 0), (2, 96, 50, 1)])
def test_particles_round_trip_in_chunks(fs, dim, nx, ny, prec):
    """More particles than the transfer scratch holds at once (no spare slots:
    capacity factor 1): what goes in comes out, values in the run's precision,
    and the fields with it; counts agree."""
    ppc = 40
    kw = dict(dim=dim, nx=nx, ny=ny, ppc=ppc, precision=prec, capacity_factor=1.0, init_plasma=0)
    rng = np.random.default_rng(nx)
    n = nx * ny * ppc
    T = np.float32 if prec else np.float64
    cell = np.arange(n) % (nx * ny)
    f = rng.random((2, n)).astype(T).astype(float)
    f[:, :3] = [0.0, 1.0 - 2.0 ** -24, 0.5]
    if dim == 1:
        f[1] = 0.0
    v = rng.normal(size=(3, n)).astype(T).astype(float)
    ids = (rng.permutation(n).astype(np.uint32) | np.where(rng.random(n) < 0.1, fs.ID_CR, 0)
           .astype(np.uint32))
    sim = fs.FauxShock(**kw)
    sim.inject(cell % nx, cell // nx, f[0], f[1], v[0], v[1], v[2], ids=ids)
    assert sim.num_particles() == n == sim.diag()["n_particles"]
    p = sim.particles()
    a, b = np.argsort(p["id"] & fs.ID_MASK), np.argsort(ids & fs.ID_MASK)
    for got, want in ((p["ci"], cell % nx), (p["cj"], cell // nx), (p["fx"], f[0]),
                      (p["fy"], f[1]), (p["vx"], v[0]), (p["vy"], v[1]), (p["vz"], v[2]),
                      (p["id"], ids)):
        np.testing.assert_array_equal(got[a], want[b])
    B = rng.normal(size=(ny, nx, 3)).astype(T).astype(float)
    sim.load_fields(B)
    np.testing.assert_array_equal(sim.grid(fs.FS_B), B)
    sim.close()


@pytest.mark.parametrize("tx,ty", [(2, 1), (2, 2), (2, 5), (3, 1), (5, 2), (3, 3), (5, 5), (10, 3)])
def test_moments_of_any_tile_shape_equal_the_oracle(fs, tx, ty):
    """The node sums with each count of candidate tiles, next to the walls and
    across the periodic rows: FP64 bit for bit, after two steps."""
    kw = dict(dim=2, nx=30, ny=30, ppc=5, dt=0.005, mach_a=12.0, theta_bn_deg=20.0, cr_enable=1,
              p_iso=40.0, seed=7)
    gpu = fs.FauxShock(tile_x=tx, tile_y=ty, **kw)
    ref = O.Oracle(**kw)
    gpu.step(2)
    ref.step(2)
    for what, name in ((fs.FS_N, O.GRID_N), (fs.FS_J, O.GRID_J), (fs.FS_B, O.GRID_B)):
        np.testing.assert_array_equal(gpu.grid(what), ref.grid(name))
    gpu.close()
    ref.close()


@pytest.mark.parametrize("scale,seed", [(1.0, 3), (1e-6, 3), (3e-23, 1), (2.5e-23, 8), (1e-25, 3)])
@pytest.mark.parametrize("prec", [0, 1])
def test_stability_number_at_any_field_strength(fs, prec, scale, seed):
    """The largest node's z, from the run's own node fields, also where the
    squares of B and u are below FP32's range: the written FP64 expression, so
    equal to rounding (a few operations of 1e-16 each)."""
    nx, ny, dt = 60, 40, 0.005
    sim = fs.FauxShock(dim=2, nx=nx, ny=ny, ppc=4, dt=dt, dx=0.5, dy=0.5, precision=prec,
                       init_plasma=0, bc_x=O.BC_PERIODIC, mach_a=0.0, beta_i=0.0, beta_e=0.0)
    rng = np.random.default_rng(seed)
    sim.load_fields(scale * rng.normal(size=(ny, nx, 3)))
    bb, n, u = sim.grid(fs.FS_BBAR), sim.grid(fs.FS_N), sim.grid(fs.FS_U)
    z = 0.5 * dt * (8.0 / 0.25 * np.sqrt((bb ** 2).sum(-1)) / n +
                    8.0 * np.sqrt((u ** 2).sum(-1)))
    assert sim.diag()["max_z"] == pytest.approx(z.max(), rel=1e-12, abs=0)
    sim.close()
