"""Routes of the demag passes and of the gradient that no other test reaches:
the chirp-z and direct passes that one-cell sides keep, the copy-engine-fed
passes on meshes that still take them, and gradients of several steps on
meshes whose forward record runs in the fused kernels.

Tolerances are the library's own (FP64 1e-12, FP32 1e-5 relative L2; 1e-4 for
an FP32 gradient against the FP64 one)."""

import numpy as np
import pytest

import workloads as wl
from oracle import micromag

torch = pytest.importorskip("torch")
import paper_2606_01114_gb300 as mm  # noqa: E402

pytestmark = pytest.mark.gpu

D = (2e-9, 2.5e-9, 3e-9)
TOL = {"f64": 1e-12, "f32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2606_01114_gb300 import build
    build.build()


def context(n, prec):
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32 if prec == "f32" else mm.MM_F64)
    mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.1, 1e5)
    return ctx


def dev(a, prec):
    return torch.tensor(a, dtype=torch.float32 if prec == "f32" else torch.float64, device="cuda")


def rel(t, ref):
    return np.linalg.norm(t.double().cpu().numpy() - ref) / np.linalg.norm(ref)


# one-cell sides: chirp-z in y, in x, direct in both; then power-of-two meshes
# of more layers than a plane block holds, whose y passes of length 512 and
# 1024 and x inverse of 512 cells are fed by the copy engine (one, some and
# many columns, a tile that is not full)
ONE_CELL = [(1, 100, 4), (1, 350, 1), (100, 1, 2), (1, 511, 16), (333, 1, 1), (1, 31, 2), (29, 1, 8)]
FED = [(8, 512, 16), (16, 256, 16), (512, 4, 16), (1, 512, 16), (2, 256, 32), (512, 256, 16)]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", ONE_CELL + FED, ids=lambda n: "x".join(map(str, n)))
def test_demag_on_the_routes_of_2n_lengths(n, prec):
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, prec)
    md = dev(m, prec)
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, micromag.Problem(n, D).demag_fft(m)) < TOL[prec]
    mm.mm_destroy(ctx)


@pytest.mark.parametrize("every", [0, 3, 7])
@pytest.mark.parametrize("n", [(64, 64, 4), (33, 61, 8), (130, 333, 2)], ids=lambda n: "x".join(map(str, n)))
def test_gradient_of_several_fused_steps(n, every):
    """Seven RK4 steps with cell-wise Ms and vacuum: the FP32 gradient, whose
    record of the steps is written by the fused kernels, against the FP64
    one."""
    rng = np.random.default_rng(sum(n))
    Ms = rng.uniform(4e5, 9e5, size=n[::-1]).astype(np.float32).astype(np.float64)
    Ms[rng.random(Ms.shape) < 0.2] = 0.0
    m = wl.random_unit(n, seed=5).astype(np.float32).astype(np.float64)
    lam0 = wl.random_unit(n, seed=6).astype(np.float32).astype(np.float64)
    out = []
    for prec in ("f64", "f32"):
        ctx = context(n, prec)
        mm.mm_set_material_fields(ctx, Ms_cell=dev(Ms, prec))
        lam = dev(lam0, prec)
        gMs = torch.zeros(ctx.shape1, dtype=lam.dtype, device="cuda")
        mm.mm_rk4_trajectory_vjp(ctx, dev(m, prec), 1e-14, 7, lam, gMs, every)
        out.append((lam.double().cpu().numpy(), gMs.double().cpu().numpy()))
        mm.mm_destroy(ctx)
    for a, b in zip(*out):
        assert np.isfinite(b).all() and np.linalg.norm(b - a) < 1e-4 * np.linalg.norm(a)


# z length 1024 in FP64: the middle level by components, one and four columns a
# block
LONG = [(5, 2, 512), (12, 6, 512), (3, 3, 512), (7, 5, 512), (2, 9, 512), (20, 17, 512), (3, 70, 512)]


@pytest.mark.parametrize("n", LONG, ids=lambda n: "x".join(map(str, n)))
def test_demag_on_the_longest_z_lines_in_double(n):
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, "f64")
    md = dev(m, "f64")
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, micromag.Problem(n, D).demag_fft(m)) < TOL["f64"]
    mm.mm_destroy(ctx)


# both sides of the lines between the fused stage and field and the kernels
# apart: one and two blocks an SM, one and two waves, x lengths of both kinds
@pytest.mark.parametrize("n", [(512, 16, 1), (512, 175, 1), (300, 200, 1), (384, 39, 1), (80, 304, 4), (80, 305, 4), (64, 351, 4),
                               (256, 83, 4), (256, 84, 4), (160, 156, 4), (160, 157, 4), (96, 234, 4), (256, 512, 8)],
                         ids=lambda n: "x".join(map(str, n)))
def test_field_and_steps_beside_the_lines(n):
    out = []
    for prec in ("f64", "f32"):
        ctx = context(n, prec)
        md = dev(wl.random_unit(n, seed=4), prec)
        H = torch.empty_like(md)
        mm.mm_effective_field(ctx, md, H)
        mm.mm_rk4_trajectory(ctx, md, 1e-14, 2)
        out.append((H.double().cpu().numpy(), md.double().cpu().numpy()))
        mm.mm_destroy(ctx)
    for a, b in zip(*out):
        assert np.linalg.norm(b - a) < TOL["f32"] * np.linalg.norm(a)


# FP64: three kernels in place of the plane kernel (few planes; z lengths 4 and
# 8, every padded y length, up to 64 cells in x) and the sizes beside the line
FEW = [(2, 100, 2), (4, 64, 2), (5, 61, 2), (8, 33, 4), (3, 32, 4), (16, 200, 2), (20, 160, 4), (33, 96, 4), (64, 256, 2),
       (64, 48, 4), (50, 190, 2), (12, 512, 4), (6, 330, 4), (64, 512, 4), (65, 64, 4), (64, 31, 2), (2, 2, 2), (2, 2, 4)]
# short x and y lengths, strips of three cells on both sides of their line
STRIPS = [(4, 3, 128), (8, 4, 1), (3, 5, 1), (3, 128, 64), (3, 256, 128), (256, 3, 64), (256, 3, 256), (3, 64, 16), (128, 3, 8)]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", FEW + STRIPS, ids=lambda n: "x".join(map(str, n)))
def test_demag_on_narrow_meshes(n, prec):
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, prec)
    md = dev(m, prec)
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, micromag.Problem(n, D).demag_fft(m)) < TOL[prec]
    mm.mm_destroy(ctx)


@pytest.mark.parametrize("n", [(2, 2, 1), (2, 4, 4), (4, 2, 2), (16, 512, 2), (32, 256, 4), (512, 128, 4), (256, 128, 4)],
                         ids=lambda n: "x".join(map(str, n)))
def test_float_float_on_narrow_and_wide_meshes(n):
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, "f64")
    mm.mm_set_fft_mode(ctx, mm.MM_FFT_FF)
    md = dev(m, "f64")
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, micromag.Problem(n, D).demag_fft(m)) < TOL["f64"]
    mm.mm_destroy(ctx)


def demag_time(n, prec):
    """Median time of one field, in us, over runs of about 5 ms."""
    ctx = context(n, prec)
    m = dev(wl.random_unit(n, seed=1), prec)
    H = torch.empty_like(m)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times, reps = [], 4
    for k in range(8):
        a.record()
        for _ in range(reps):
            mm.mm_demag_field(ctx, m, H)
        b.record()
        torch.cuda.synchronize()
        us = a.elapsed_time(b) * 1e3 / reps
        if k < 3:
            reps = max(2, min(200, int(5e3 / us)))
        else:
            times.append(us)
    mm.mm_destroy(ctx)
    return sorted(times)[len(times) // 2]


# (narrow mesh, wider mesh, share of its time): an eighth of the columns may cost
# half; three cells may cost what four do
@pytest.mark.parametrize("prec,n,wide,share", [
    ("f64", (16, 512, 4), (128, 512, 4), 0.5), ("f64", (2, 256, 4), (128, 256, 4), 0.5), ("f64", (3, 512, 512), (4, 512, 512), 1.05),
    ("f64", (512, 3, 256), (512, 4, 256), 1.05), ("f32", (512, 3, 512), (512, 4, 512), 1.05)])
def test_a_narrow_mesh_costs_less_than_a_wide_one(prec, n, wide, share):
    assert demag_time(n, prec) < share * demag_time(wide, prec)
