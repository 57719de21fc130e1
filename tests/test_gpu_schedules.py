"""Schedules of the demag convolution chosen by grid size, against the
size-generic passes (which the oracle checks in test_gpu_parity.py).

Tolerance: a schedule's field has about one FP32 rounding (6e-8 relative) per
radix pass, at most 11 passes per axis and direction, so 66 in all, adding up
in quadrature to 5e-7 of the field's norm; two schedules then differ by 7e-7.
2e-6 leaves a factor of three.
"""
import numpy as np
import pytest
import torch

from helpers import cfg_of, context, random_m, rel_l2

pytestmark = pytest.mark.gpu

TOL = 2e-6


def field(c, **kw):
    from paper_2602_12242_gb300 import MX_TERM_DEMAG
    from paper_2602_12242_gb300.solver import from_dev4, to_dev4
    ctx = context(c, **kw)
    h = from_dev4(ctx.heff(to_dev4(np.asarray(random_m(c, 41), np.float32)), terms=MX_TERM_DEMAG))
    ctx.sync()
    return h, ctx


# (nx, ny, nz): Py/2 = 16 .. 256 with Pz = 4 .. 32, full and ragged nz <= Pz/2 and ny <= Py/2,
# one and two kx columns per block (Hx above and below 608), an odd last column
FEW_LAYERS = [(40, 9, 2), (33, 16, 16), (20, 13, 9), (64, 32, 16), (37, 21, 5), (30, 17, 13), (50, 64, 8), (40, 40, 4),
              (41, 33, 2), (70, 128, 5), (24, 100, 4), (30, 77, 2), (20, 65, 7), (24, 256, 2), (600, 24, 2),
              (1000, 10, 3), (513, 33, 4)]


@pytest.mark.parametrize("shape", FEW_LAYERS)
def test_few_layer_kernel_matches_generic_passes(shape):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx = field(c)
    assert ctx.kernel_name("yz_fused") == "yz3_kernel"
    ref, _ = field(c, demag_path=_lib.MX_DEMAG_GENERIC)
    assert rel_l2(h, ref) <= TOL


# (nx, ny, nz): Pz/2 = 16 .. 512 and Py/2 = 16 .. 512, full and ragged depths, a last kx tile of one
# column (Hx = 65) and of part of one
DEEP = [(40, 33, 64), (33, 64, 33), (20, 100, 16), (50, 20, 100), (24, 17, 129), (64, 65, 40), (17, 130, 30),
        (16, 300, 20), (30, 12, 260), (20, 257, 17), (40, 40, 20), (100, 9, 65)]


@pytest.mark.parametrize("shape", DEEP)
def test_deep_grid_kernels_match_generic_passes(shape):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx = field(c)
    assert ctx.kernel_name("z_mul") == ("deep_z3_kernel" if ctx.padded_dims[2] > 128 else "deep_z_kernel")
    ref, gen = field(c, demag_path=_lib.MX_DEMAG_GENERIC)
    assert gen.kernel_name("z_mul") == "z_mul_kernel"
    assert rel_l2(h, ref) <= TOL
    # the stored tensor spectrum reads back in the documented order
    assert torch.equal(ctx.demag_spectrum(), gen.demag_spectrum())


# (nx, ny, nz) with many rows: every row length Px/2 = 16 .. 1024 of the many-row x kernels, odd nx,
# a last block of part of its rows
ROWS = [(9, 101, 99), (17, 100, 101), (33, 70, 60), (127, 61, 43), (129, 41, 33), (300, 37, 35), (520, 33, 31)]


@pytest.mark.parametrize("shape", ROWS)
@pytest.mark.parametrize("ms_map", [False, True])
def test_many_row_x_kernels_match_generic_passes(shape, ms_map):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    Ms = np.random.default_rng(43).uniform(6e5, 1e6, size=shape[::-1]) if ms_map else None
    h, ctx = field(c, Ms=Ms)
    assert (ctx.kernel_name("x_fwd"), ctx.kernel_name("x_inv")) == ("xf_many_kernel", "xi_many_kernel")
    ref, gen = field(c, Ms=Ms, demag_path=_lib.MX_DEMAG_GENERIC)
    assert gen.kernel_name("x_fwd") == "x_fwd_kernel"
    assert rel_l2(h, ref) <= TOL


# (nx, ny): one layer, Px/2 and Py/2 = 16 .. 1024 and 16 .. 512, one, two and four columns per
# block and the wide kernel, odd last columns, ragged rows
FILMS = [(9, 9), (16, 16), (31, 30), (70, 20), (640, 30), (33, 33), (200, 60), (700, 50), (100, 100), (300, 128),
         (1000, 70), (60, 200), (200, 150), (300, 200), (120, 300), (130, 500)]


@pytest.mark.parametrize("shape", FILMS)
def test_film_kernels_match_generic_passes(shape):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=shape[0], ny=shape[1], nz=1, dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx = field(c)
    wide = (shape[1] > 256 and shape[0] > 128) or (128 < shape[1] <= 256 and shape[0] > 256)
    assert ctx.kernel_name("yz_fused") == ("yz2d_wide_kernel" if wide else "yz2d_kernel")
    ref, _ = field(c, demag_path=_lib.MX_DEMAG_GENERIC)
    assert rel_l2(h, ref) <= TOL


@pytest.mark.parametrize("shape", [(9, 9, 1), (31, 30, 1), (40, 20, 3), (65, 33, 1), (200, 60, 2), (300, 40, 1),
                                   (1000, 33, 1)])
@pytest.mark.parametrize("ms_map", [False, True])
def test_row_kernel_steps_match_generic_passes(shape, ms_map):
    """Every row length, ragged, with DMI: two RK4 steps (the four stages' updates, and the rows that a
    step leaves transformed for the next) against the separate kernels on the generic passes."""
    from paper_2602_12242_gb300 import _lib
    from paper_2602_12242_gb300.solver import from_dev4, to_dev4
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9, D=1e-3, dmi=True)
    Ms = np.random.default_rng(47).uniform(6e5, 1e6, size=shape[::-1]) if ms_map else None
    out = []
    for kw in ({}, dict(demag_path=_lib.MX_DEMAG_GENERIC)):
        ctx = context(c, Ms=Ms, **kw)
        m = to_dev4(np.asarray(random_m(c, 48), np.float32))
        ctx.rk_step(m, 2, 1e-14, "rk4")
        out.append(from_dev4(m))
        name = ctx.kernel_name("x_inv_local")
        assert name == ("xr_kernel" if not kw else "")
    assert rel_l2(out[0], out[1]) <= TOL


@pytest.mark.parametrize("shape", [(40, 20, 1), (33, 16, 3), (40, 33, 64), (64, 64, 16)])
@pytest.mark.parametrize("n", [2, 3, 4])
def test_euler_step_pairs_equal_single_steps(shape, n):
    """Row-kernel, deep and plane grids: a call of n steps (pairs of steps and the odd one) against n
    calls of one step, also when the two kinds of call alternate.  A call renormalises m first, which
    changes a component by a few FP32 roundings (6e-8) per call."""
    from paper_2602_12242_gb300.solver import from_dev4, to_dev4
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    ctx = context(c)
    m0 = np.asarray(random_m(c, 49), np.float32)
    a, b = to_dev4(m0), to_dev4(m0)
    for _ in range(2):
        ctx.rk_step(a, n, 1e-14, "euler")
        ctx.rk_step(a, 1, 1e-14, "euler")
    for _ in range(2 * (n + 1)):
        ctx.rk_step(b, 1, 1e-14, "euler")
    assert np.abs(from_dev4(a) - from_dev4(b)).max() <= 2e-6


# (nx, ny, nz, kernel): 65 kx columns on the plane path, both sides of the line between the four-CTA and
# the few-layer kernel, and 129 columns
@pytest.mark.parametrize("nx,ny,nz,kernel", [
    (33, 128, 8, "yzq_kernel"), (64, 65, 5, "yzq_kernel"), (50, 200, 5, "yzq_kernel"), (40, 300, 3, "yzq_kernel"),
    (50, 140, 4, "yz3_kernel"), (33, 300, 2, "yz3_kernel"), (64, 64, 9, "yz3_kernel"), (65, 128, 8, "yz3_kernel")])
def test_plane_kernel_of_few_columns(nx, ny, nz, kernel):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=nx, ny=ny, nz=nz, dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx = field(c)
    assert (ctx.kernel_name("x_fwd"), ctx.kernel_name("yz_fused")) == ("xfk_kernel", kernel)
    ref, _ = field(c, demag_path=_lib.MX_DEMAG_GENERIC)
    assert rel_l2(h, ref) <= TOL


@pytest.mark.parametrize("path,nx,ny,nz,fewer,kernel", [
    ("MX_DEMAG_AUTO", 40, 512, 16, 9, "yzq_kernel"), ("MX_DEMAG_AUTO", 64, 128, 8, 5, "yzq_kernel"),
    ("MX_DEMAG_PLANE_PAIR", 64, 200, 4, 3, "yzh_kernel"), ("MX_DEMAG_PLANE", 40, 32, 16, 9, "yzh_kernel")])
def test_a_newer_context_of_fewer_layers_leaves_the_older_one_usable(path, nx, ny, nz, fewer, kernel):
    """Both contexts launch the same kernel, the older one with more shared memory."""
    from paper_2602_12242_gb300 import MX_TERM_DEMAG, _lib
    from paper_2602_12242_gb300.solver import to_dev4
    ctx = [None, None]
    c = cfg_of(nx=nx, ny=ny, nz=nz, dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx[0] = field(c, demag_path=getattr(_lib, path))
    _, ctx[1] = field(dict(c, nz=fewer), demag_path=getattr(_lib, path))
    assert [x.kernel_name("yz_fused") for x in ctx] == [kernel, kernel]
    again = ctx[0].heff(to_dev4(np.asarray(random_m(c, 41), np.float32)), terms=MX_TERM_DEMAG)
    ctx[0].sync()
    assert np.array_equal(again[..., :3].cpu().numpy(), h.astype(np.float32))


@pytest.mark.parametrize("shape,path", [((40, 20, 1), "MX_DEMAG_AUTO"), ((40, 33, 64), "MX_DEMAG_AUTO"),
                                        ((64, 64, 9), "MX_DEMAG_PLANE"), ((64, 64, 9), "MX_DEMAG_PLANE_XLOCAL")])
@pytest.mark.parametrize("n", [1, 4, 5])
def test_profile_times_the_euler_steps_of_a_run(shape, path, n):
    """The copy that ends a single Euler step is timed for the odd step of a run only, and the profiled
    steps give the run's bits."""
    from paper_2602_12242_gb300 import _lib
    from paper_2602_12242_gb300.solver import to_dev4
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    ctx = context(c, demag_path=getattr(_lib, path))
    m0 = np.asarray(random_m(c, 50), np.float32)
    a, b = to_dev4(m0), to_dev4(m0)
    ctx.rk_step(a, n, 1e-14, "euler")
    prof = ctx.profile_step(b, n, 1e-14, "euler")
    assert prof.get("copy", (0.0, 0))[1] == n % 2
    assert torch.equal(a, b)


# (nx, ny, nz, kx-major): every (Py/2, Pz) that the few-layer kernel runs on the plane path's layout, and
# those of long columns and of two kx columns per block (Hx > 608) in place
@pytest.mark.parametrize("nx,ny,nz,km", [
    (100, 50, 14, True), (64, 64, 16, True), (100, 128, 8, True), (40, 150, 4, True), (100, 256, 3, True),
    (100, 150, 6, True), (70, 256, 8, True), (40, 300, 2, True), (100, 512, 2, True), (100, 280, 3, True),
    (20, 50, 14, False), (30, 100, 7, False), (20, 200, 4, False), (24, 256, 3, False), (20, 150, 6, False),
    (24, 256, 8, False), (20, 300, 2, False), (24, 512, 2, False), (20, 280, 3, False),
    (1000, 60, 4, False), (600, 100, 3, False), (600, 200, 2, False), (600, 60, 7, False), (600, 30, 14, False),
    (1000, 12, 15, False), (520, 9, 7, False)])
def test_few_layer_kernel_of_every_layout_matches_generic_passes(nx, ny, nz, km):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=nx, ny=ny, nz=nz, dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx = field(c)
    assert ctx.kernel_name("yz_fused") == "yz3_kernel"
    assert (ctx.kernel_name("x_fwd") == "xfk_kernel") == km
    ref, _ = field(c, demag_path=_lib.MX_DEMAG_GENERIC)
    assert rel_l2(h, ref) <= TOL


# films of 2049 kx columns: eight columns per block (rows of up to 64), four, and the wide kernel, after the
# size-generic x passes
@pytest.mark.parametrize("nx,ny", [(1025, 16), (1300, 9), (1100, 30), (1025, 60), (1100, 100), (1030, 130), (1025, 257)])
def test_film_kernels_of_many_columns_match_generic_passes(nx, ny):
    from paper_2602_12242_gb300 import _lib
    c = cfg_of(nx=nx, ny=ny, nz=1, dx=2e-9, dy=2.5e-9, dz=3e-9)
    h, ctx = field(c)
    assert ctx.padded_dims[0] == 4096 and ctx.kernel_name("x_fwd") == "x_fwd_kernel"
    assert ctx.kernel_name("yz_fused") == ("yz2d_wide_kernel" if ny > 128 else "yz2d_kernel")
    ref, _ = field(c, demag_path=_lib.MX_DEMAG_GENERIC)
    assert rel_l2(h, ref) <= TOL


# Deep grids whose row kernels are at most a block per SM, so that the y pass starts while they run: one
# field after another and steps, against the generic passes.  (The spectrum of the field or stage before
# is an error of order one in H, 1e-3 of m per step here.)
@pytest.mark.parametrize("shape", [(26, 25, 20), (28, 24, 25), (64, 17, 17), (12, 20, 25), (16, 33, 18), (40, 17, 17)])
def test_deep_grids_of_few_rows_match_generic_passes(shape):
    from paper_2602_12242_gb300 import MX_TERM_DEMAG, _lib
    from paper_2602_12242_gb300.solver import from_dev4, to_dev4
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    ms = [to_dev4(np.asarray(random_m(c, q), np.float32)) for q in (41, 42, 43)]
    out = []
    for path in (_lib.MX_DEMAG_AUTO, _lib.MX_DEMAG_GENERIC):
        ctx = context(c, demag_path=path)
        if path == _lib.MX_DEMAG_AUTO:
            assert ctx.kernel_name("y_fwd") == "deep_yf_kernel" and ctx.kernel_name("x_inv_local") == "xr_kernel"
        got = []
        for _ in range(3):
            got += [ctx.heff(m, terms=MX_TERM_DEMAG) for m in ms] + [ctx.llg_rhs(m) for m in ms]
        for method in ("rk4", "euler"):
            for n in (2, 5):
                m = ms[0].clone()
                ctx.rk_step(m, n, 1e-14, method)
                got.append(m)
        ctx.sync()
        out.append([from_dev4(x) for x in got])
    for a, b in zip(*out):
        assert rel_l2(a, b) <= TOL


# Few-layer and one-layer grids of at most a block per SM in every kernel: the inverse x pass, on both
# layouts of the spectrum, starts while the y/z kernel runs, and the right-hand side's local kernel while
# the inverse x pass does
@pytest.mark.parametrize("shape", [(100, 128, 5), (50, 64, 14), (60, 100, 4), (40, 20, 2), (20, 30, 1), (100, 16, 9)])
def test_short_chains_of_fields_match_generic_passes(shape):
    from paper_2602_12242_gb300 import MX_TERM_DEMAG, _lib
    from paper_2602_12242_gb300.solver import from_dev4, to_dev4
    c = cfg_of(nx=shape[0], ny=shape[1], nz=shape[2], dx=2e-9, dy=2.5e-9, dz=3e-9)
    ms = [to_dev4(np.asarray(random_m(c, q), np.float32)) for q in (41, 42, 43)]
    out = []
    for path in (_lib.MX_DEMAG_AUTO, _lib.MX_DEMAG_GENERIC):
        ctx = context(c, demag_path=path)
        got = []
        for _ in range(3):
            got += [ctx.heff(m, terms=MX_TERM_DEMAG) for m in ms] + [ctx.llg_rhs(m) for m in ms]
        ctx.sync()
        out.append([from_dev4(x) for x in got])
    for a, b in zip(*out):
        assert rel_l2(a, b) <= TOL
