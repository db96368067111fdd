"""Values at the ends of the types' ranges, runs with an error pending, and
several live handles of one kernel: each against the written expressions, or
against the same calls made alone."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle as O
from tests import window_inputs as WI
from tests import workloads as W

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


@pytest.mark.parametrize("scale,seed,n_floor,dx,n_part", [
    (3e-23, 1, 1e-20, 0.5, 0), (2.5e-23, 8, 1e-18, 0.5, 0), (1e-22, 3, 1e-20, 0.5, 0),
    (3e-23, 4, 0.05, 1e-8, 0), (2e-23, 6, 0.05, 1e-9, 600), (1e-20, 5, 1e-30, 0.5, 0),
    (1.0, 2, 1e-25, 0.5, 600), (1e-15, 7, 1e-12, 1e-3, 600)])
@pytest.mark.parametrize("prec", [0, 1])
def test_stability_number_of_thin_plasma_and_small_cells(fs, prec, scale, seed, n_floor, dx, n_part):
    """The largest node's z where it is not small although the squares of B (or
    u) are below FP32's range, by 1/n or 1/dx^2: the written FP64 expression on
    the run's own node fields, so equal to rounding."""
    nx, ny, dt = 60, 40, 0.005
    sim = fs.FauxShock(dim=2, nx=nx, ny=ny, ppc=4, dt=dt, dx=dx, dy=dx, precision=prec,
                       init_plasma=0, bc_x=O.BC_PERIODIC, mach_a=0.0, beta_i=0.0, beta_e=0.0,
                       n_floor=n_floor)
    rng = np.random.default_rng(seed)
    if n_part:
        p = list(W.random_particles(rng, n_part, nx, ny))
        sim.inject(*p[:4], *[scale * v for v in p[4:]])
    sim.load_fields(scale * rng.normal(size=(ny, nx, 3)))
    bb, n, u = sim.grid(fs.FS_BBAR), sim.grid(fs.FS_N), sim.grid(fs.FS_U)
    z = 0.5 * dt * (8.0 / dx ** 2 * np.sqrt((bb ** 2).sum(-1)) / n +
                    4.0 / dx * np.sqrt((u ** 2).sum(-1)))
    assert sim.diag()["max_z"] == pytest.approx(z.max(), rel=1e-12, abs=0)
    sim.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_stability_number_passes_over_nan_nodes(fs, prec):
    """A node without a z (NaN field) next to fast plasma: the largest of the rest."""
    nx, ny = 60, 40
    sim = fs.FauxShock(dim=2, nx=nx, ny=ny, ppc=4, precision=prec, init_plasma=0,
                       bc_x=O.BC_PERIODIC, mach_a=0.0, beta_i=0.0, beta_e=0.0)
    rng = np.random.default_rng(9)
    p = list(W.random_particles(rng, 600, nx, ny))
    p[4][:50] += 1e4
    p[0][:50], p[1][:50] = 10, 10
    sim.inject(*p)
    B = rng.normal(size=(ny, nx, 3))
    B[8:13, 8:13] = np.nan
    sim.load_fields(B)
    bb, n, u = sim.grid(fs.FS_BBAR), sim.grid(fs.FS_N), sim.grid(fs.FS_U)
    z = 0.0025 * (32.0 * np.sqrt((bb ** 2).sum(-1)) / n + 8.0 * np.sqrt((u ** 2).sum(-1)))
    assert np.isnan(z[10, 10]) and u[10, 10, 0] > 100 * np.nanmax(z)
    assert sim.diag()["max_z"] == pytest.approx(np.nanmax(z), rel=1e-12, abs=0)
    sim.close()


def test_energy_and_momentum_of_subnormal_velocities(fs):
    """FP32 velocities below the normal range count in the sums with their exact
    values (FP64 sums of some hundred terms)."""
    nx, n = 32, 300
    sim = fs.FauxShock(dim=1, nx=nx, ppc=4, precision=1, init_plasma=0, bc_x=O.BC_PERIODIC,
                       mach_a=0.0, beta_i=0.0, beta_e=0.0, capacity_factor=16.0)
    rng = np.random.default_rng(1)
    v = rng.choice([1e-45, 3e-42, 1e-40, 1.1e-38, 2e-38, 0.0], (3, n)) * rng.choice([-1, 1], (3, n))
    sim.inject(rng.integers(0, nx, n), np.zeros(n), rng.random(n), np.zeros(n), *v)
    p, d = sim.particles(), sim.diag()
    w = 0.25 * 0.5
    for k in ("vx", "vy", "vz"):
        assert np.abs(p[k]).min() < 1e-44 < np.abs(p[k]).max()
        assert d["p" + k[1]] == pytest.approx((w * p[k]).sum(), rel=1e-9, abs=0)
    e = (0.5 * w * (p["vx"] ** 2 + p["vy"] ** 2 + p["vz"] ** 2)).sum()
    assert d["kinetic"] == pytest.approx(e, rel=1e-12, abs=0)
    sim.close()


@pytest.mark.parametrize("dim,chain", [(1, 10), (2, 20)])
def test_fp32_deposit_adds_short_chains(fs, dim, chain):
    """160 equal particles at rest in one cell: their FP32 sum errs no more than
    sums of `chain` terms, added in pairs (exact, the sums being equal), would.
    With these offsets a chain of twice that errs at least twice as much."""
    f = 0.5 - 7.0 * 2.0 ** -24
    n, cell = 160, 3
    sim = fs.FauxShock(dim=dim, nx=8, ny=4 if dim == 2 else 1, ppc=64, precision=1, init_plasma=0,
                       bc_x=O.BC_PERIODIC, mach_a=0.0, beta_i=0.0, beta_e=0.0, n_floor=1e-6,
                       tile_x=2, capacity_factor=8.0)
    z = np.zeros(n)
    sim.inject(np.full(n, cell), z, np.full(n, f), z, z, z, z)
    sim.step(1)
    got = sim.grid(fs.FS_N)[0]

    def err(x, terms):
        s = np.float32(0)
        for _ in range(terms):
            s = np.float32(s + np.float32(x))
        return abs(float(s) / (terms * float(np.float32(x))) - 1)
    for node, x in ((cell, 1.0 - f), (cell + 1, f)):
        allowed = err(x, chain)
        assert err(x, 2 * chain) > 2 * allowed
        assert abs(got[node] / (n / 64 * x) - 1) <= allowed * (1 + 1e-6)
    sim.close()


def window(fs, prec, n_sub, steps, ckpt, nx=64):
    from paper_2507_14282_gb300 import window as m
    X, V = WI.plasma(nx, 8)
    amps, ph = WI.modes()
    w = m.FauxShockWindow(X, V, ph, steps=steps, ckpt=ckpt, nx=nx, ny=1, ppc=8, n_sub=n_sub,
                          precision=prec, cr_enable=1, fs_mode_thermal=1, p_iso=100.0,
                          n_cr_ratio=0.01, **WI.COMMON)
    return w, WI.theta(amps)


# A window run twice: the forward's sums are fixed point, so the loss repeats
# exactly; the backward adds in FP64 in any order, and an FP32 adjoint rounds
# what came out, at some 1e-7 of its size.
GRAD_REPEATS = {0: 1e-11, 1: 1e-5}


@pytest.mark.parametrize("prec,n_sub", [(0, 9), (1, 10)])
def test_window_runs_on_after_one_of_fewer_substeps(fs, prec, n_sub):
    """A live window keeps its kernels' shared memory when a later one needs less."""
    first, th = window(fs, prec, n_sub, 6, 3)
    L, g = first.loss_and_grad(th)
    second, _ = window(fs, prec, 2, 6, 3)
    second.loss_and_grad(th)
    again = first.loss_and_grad(th)
    assert again[0] == L
    np.testing.assert_allclose(again[1], g, rtol=0, atol=GRAD_REPEATS[prec] * np.abs(g).max())
    first.close()
    second.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_batch_runs_on_after_one_of_narrower_tiles(fs, prec):
    """The same for the batched push: the second batch's tiles need less."""
    kw = dict(dim=1, nx=256, ppc=8, precision=prec, mach_a=10.0, dt=0.005, capacity_factor=8.0)
    alone = fs.FauxShock(tile_x=64, **kw)
    wide = [fs.FauxShock(tile_x=64, **kw) for _ in range(2)]
    narrow = [fs.FauxShock(tile_x=2, **kw) for _ in range(2)]
    batches = [fs.FsBatch(wide), fs.FsBatch(narrow)]
    alone.step(3)
    for b in batches[::-1]:
        b.step(1)
        b.step(2)
    for s in wide:
        assert s.diag()["step"] == 3
        np.testing.assert_allclose(s.grid(fs.FS_B), alone.grid(fs.FS_B), rtol=0,
                                   atol=1e-4 if prec else 0)
    for b in batches:
        b.close()
    for s in [alone] + wide + narrow:
        s.close()


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("what", ["B", "N", "PROFILE_N", "PROFILE_DB2", "PROFILE_B",
                                  "SPECTRUM_BPERP", "SPECTRUM_P_ALL", "HIST_XPX", "STATE"])
@pytest.mark.parametrize("on_device", [0, 1])
def test_reads_of_a_run_with_an_error_pending_leave_their_destination(fs, dim, what, on_device):
    """A non-finite motion that only the device knows of yet: its code comes back,
    also from a read that is refused for its size, and nothing is written."""
    import torch
    cfg = W.scaled(W.CONFIG_2D if dim == 2 else W.CONFIG_1D, nx=64, ppc=8,
                   **(dict(ny=16) if dim == 2 else {}))
    for size in (1 << 20, 4):
        sim = fs.FauxShock(precision=0, **cfg)
        B = sim.grid(fs.FS_B)
        B[0, 20, 1] = np.nan
        sim.load_fields(B)
        sim.step(1)
        dst = torch.full((1 << 20,), 7, dtype=torch.uint8, device="cuda" if on_device else "cpu")
        torch.cuda.synchronize()
        rc = fs.lib().fs_moments(sim._h, getattr(fs, "FS_" + what), C.c_void_p(dst.data_ptr()),
                                 C.c_size_t(size), on_device)
        torch.cuda.synchronize()
        assert rc == fs.FS_ENAN
        assert bool((dst == 7).all())
        sim.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("steps,ckpts", [(23, (1, 2, 5, 8, 22)), (24, (3, 12))])
def test_window_segments_of_any_length_give_one_gradient(fs, prec, steps, ckpts):
    """One tape for all segments, a segment written into it while the one after it
    is read back: against the same window in one segment."""
    whole, th = window(fs, prec, 2, steps, steps)
    L, g = whole.loss_and_grad(th)
    for ckpt in ckpts:
        w, _ = window(fs, prec, 2, steps, ckpt)
        for _ in range(3):
            L1, g1 = w.loss_and_grad(th)
            assert L1 == L
            np.testing.assert_allclose(g1, g, rtol=0, atol=GRAD_REPEATS[prec] * np.abs(g).max())
        w.close()
    whole.close()
