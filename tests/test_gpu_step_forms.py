"""The step's kernels at the edges of their splits, against the oracle: the 2D
field marches at their strips' edges, the 1D field launch's two alternating
buffers, long deposit runs and weights that are no power of two, many injected
particles, and a window whose slots are in no order of their cells. FP64 bit for
bit; FP32 within the bound of one step of the precision form (relative L2 1e-5)."""
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


def pair(fs, precision, **cfg):
    gpu = fs.FauxShock(precision=precision, **cfg)
    ref = O.Oracle(**{k: v for k, v in cfg.items()
                      if k not in ("tile_x", "tile_y", "capacity_factor")})
    return gpu, ref


def compare(fs, gpu, ref, exact):
    for what, name in ((fs.FS_B, O.GRID_B), (fs.FS_E, O.GRID_E), (fs.FS_N, O.GRID_N),
                       (fs.FS_U, O.GRID_U), (fs.FS_J, O.GRID_J)):
        a, b = gpu.grid(what), ref.grid(name)
        if exact:
            np.testing.assert_array_equal(a, b)
        else:
            assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b), what


# a strip of nodes holds 30 columns in FP64; 23 in FP32, 22 in the last substep
@pytest.mark.parametrize("prec,nx,ny,n_sub", [
    (0, 28, 3, 1), (0, 29, 3, 1), (0, 30, 2, 2), (0, 31, 41, 3), (0, 60, 5, 2), (0, 2, 16, 1),
    (1, 21, 4, 1), (1, 22, 9, 2), (1, 23, 3, 3), (1, 44, 11, 2), (1, 46, 33, 1), (1, 4, 2, 2)])
@pytest.mark.parametrize("bc", ["walls", "periodic"])
def test_field_march_strip_edges(fs, prec, nx, ny, n_sub, bc):
    cfg = W.scaled(W.CONFIG_2D_FP32 if prec else W.CONFIG_2D, nx=nx, ny=ny, ppc=16, n_sub=n_sub,
                   theta_bn_deg=30.0, tile_x=next(t for t in range(2, nx + 1) if nx % t == 0),
                   tile_y=1, capacity_factor=8.0)
    if bc == "periodic":
        cfg.update(bc_x=O.BC_PERIODIC, mach_a=1.0, j_cr_ext=0.2)
    gpu, ref = pair(fs, prec, **cfg)
    for steps in (1,) if prec else (1, 3):
        gpu.step(steps)
        ref.step(steps)
        compare(fs, gpu, ref, not prec)
    gpu.close()
    ref.close()


@pytest.mark.parametrize("nx,n_sub", [(31, 2), (32, 1), (33, 16), (96, 2), (64, 17)])
def test_alternating_field_buffers_1d(fs, nx, n_sub):
    """Odd step counts, then particles put in, then fields: each acts on the
    buffers of the step that comes next."""
    cfg = W.scaled(W.CONFIG_1D, nx=nx, ppc=8, n_sub=n_sub, capacity_factor=16.0,
                   tile_x=next(t for t in range(2, nx + 1) if nx % t == 0))
    gpu, ref = pair(fs, 0, **cfg)
    rng = np.random.default_rng(nx)
    for steps in (1, 2, 3):
        gpu.step(steps)
        ref.step(steps)
        compare(fs, gpu, ref, True)
        new = W.random_particles(rng, 5, nx, 1)
        gpu.inject(*new)
        ref.inject(*new)
        gpu.step(1)
        ref.step(1)
        compare(fs, gpu, ref, True)
        B = ref.grid(O.GRID_B) * 1.01
        gpu.load_fields(B)
        ref.set_B(B)
    gpu.step(5)
    ref.step(5)
    compare(fs, gpu, ref, True)
    gpu.close()
    ref.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("dim,ppc,tile", [(1, 161, 2), (1, 512, 2), (2, 160, 2), (2, 700, 2),
                                          (2, 24, 4), (2, 1, 4)])
def test_deposit_runs_and_weights(fs, prec, dim, ppc, tile):
    """Cells of more particles than one piece of the deposit (160) and than one
    chunk, with weights that are powers of two and that are not, both species."""
    cfg = dict(dim=dim, nx=8, ny=4 if dim == 2 else 1, ppc=ppc, dt=0.005, mach_a=12.0,
               theta_bn_deg=20.0, cr_enable=1, p_iso=40.0, n_cr_ratio=0.0125, seed=7, tile_x=tile,
               capacity_factor=8.0)
    gpu, ref = pair(fs, prec, **cfg)
    for steps in (1,) if prec else (1, 4):
        gpu.step(steps)
        ref.step(steps)
        compare(fs, gpu, ref, not prec)
    gpu.close()
    ref.close()


@pytest.mark.parametrize("ny,ppc", [(1, 64), (60, 64), (64, 400), (300, 4)])
def test_many_injected_particles(fs, ny, ppc):
    """Few particles a step (one block counts and draws) and many (a count and
    a grid of draws), more rows than a block too."""
    cfg = dict(dim=2 if ny > 1 else 1, nx=8, ny=ny, ppc=ppc, dt=0.01, mach_a=30.0,
               theta_bn_deg=20.0, cr_enable=1, p_iso=40.0, seed=7, tile_x=2, capacity_factor=8.0)
    gpu, ref = pair(fs, 0, **cfg)
    gpu.step(4)
    ref.step(4)
    compare(fs, gpu, ref, True)
    assert gpu.diag()["injected"] == ref.diag()["injected"] > 0
    gpu.close()
    ref.close()


@pytest.mark.parametrize("ckpt", [7, 100])
def test_window_slots_in_any_order_match_the_oracle(fs, ckpt):
    """Slots whose cells span more than a block's sort takes (64), in several
    segments and in one. The bounds are those of the ordered window."""
    from oracle import window as wo
    from paper_2507_14282_gb300 import window as fsw
    nx = 100
    X, V = WI.plasma(nx, 8)
    mix = np.random.default_rng(1).permutation(X.size)
    X, V = X[mix], V[mix]
    amps, ph = WI.modes()
    th = WI.theta(amps)
    spec = wo.WindowSpec(nx=nx, ppc=8, X0=X, V0=V, phases=ph, **WI.COMMON)
    L0, g0, win = wo.loss_and_grad(spec, th, 100)
    w = fsw.FauxShockWindow(X, V, ph, steps=100, ckpt=ckpt, nx=nx, ny=1, ppc=8, precision=0,
                            cr_enable=1, fs_mode_thermal=1, p_iso=100.0, n_cr_ratio=0.01,
                            **WI.COMMON)
    L, g = w.loss_and_grad(th)
    assert w.counts() == win.counts
    assert L == pytest.approx(L0, rel=1e-9)
    gm = np.abs(g0[:16]).max()
    np.testing.assert_allclose(g[:16], g0[:16], rtol=0, atol=1e-6 * gm)
    assert g[16] == pytest.approx(g0[16], rel=1e-5)
    assert g[17] == pytest.approx(g0[17], rel=1e-6)
    w.close()


def march_rows(strips, ny, extra, lo, hi):
    """Rows of a warp's march, as the launcher chooses them for 152 SMs."""
    rows, best = 1, -1
    for r in range(1, min(128, ny) + 1):
        per_sm = (strips * -(-ny // r) + 151) // 152
        if best >= 0 and per_sm < lo:
            break
        cost = per_sm * (r + extra)
        if best >= 0 and cost >= best and per_sm <= hi:
            continue
        best = -1 if per_sm > hi else cost
        rows = r
    return rows


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("nx,ny,n_sub", [(1002, 152, 1), (1002, 152, 2), (1024, 256, 3)])
@pytest.mark.parametrize("bc", ["walls", "periodic"])
def test_field_march_of_several_rows(fs, prec, nx, ny, n_sub, bc):
    """Marches that carry a row's sums to the next, with a short last march."""
    for cols, extra, lo in ((23, 9, 8), (22, 10, 8)) if prec else ((30, 2, 11),):
        rows = march_rows(-(-(nx + (bc == "walls")) // cols), ny, extra, lo, 16)
        assert rows > 1 and ny % rows
    cfg = W.scaled(W.CONFIG_2D_FP32 if prec else W.CONFIG_2D, nx=nx, ny=ny, ppc=2, n_sub=n_sub,
                   theta_bn_deg=30.0)
    if bc == "periodic":
        cfg.update(bc_x=O.BC_PERIODIC, mach_a=1.0, j_cr_ext=0.2)
    gpu, ref = pair(fs, prec, **cfg)
    gpu.step(1)
    ref.step(1)
    compare(fs, gpu, ref, not prec)
    gpu.close()
    ref.close()


@pytest.mark.parametrize("first", [1, 3])
def test_runs_changed_after_an_odd_number_of_batched_steps(fs, first):
    """Particles put in and fields loaded between odd numbers of batched steps act
    on the buffers of the step that comes next."""
    cfgs = [W.scaled(W.CONFIG_1D, nx=nx, ppc=8, seed=nx, capacity_factor=16.0) for nx in (64, 96, 256)]
    runs = [pair(fs, 0, **c) for c in cfgs]
    batch = fs.FsBatch([g for g, _ in runs])
    for steps in (first, 2, 1):
        batch.step(steps)
        for k, (gpu, ref) in enumerate(runs):
            ref.step(steps)
            compare(fs, gpu, ref, True)
            new = W.random_particles(np.random.default_rng(steps + k), 5, cfgs[k]["nx"], 1)
            gpu.inject(*new)
            ref.inject(*new)
            compare(fs, gpu, ref, True)
        batch.step(1)
        for gpu, ref in runs:
            ref.step(1)
            compare(fs, gpu, ref, True)
            B = ref.grid(O.GRID_B) * 1.01
            gpu.load_fields(B)
            ref.set_B(B)
    batch.step(2)
    for gpu, ref in runs:
        ref.step(2)
        compare(fs, gpu, ref, True)
    batch.close()
    for gpu, ref in runs:
        gpu.close()
        ref.close()
