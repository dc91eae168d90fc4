"""The plane-layout demag passes (spectra stored per kx plane, lengths padded
to {4, 5, 6, 8} 2^k) against the float64 oracle: every padded y length of the
table with its neighbours, both routes (one block per plane, and y / z / y as
three kernels), odd sides, the smallest sides, per-cell Ms with vacuum, the
Ms = 1 operator of the adjoint, and the float-float kernels.

Tolerances are the library's own per precision (FP64 and float-float 1e-12,
FP32 1e-5 relative L2), set before the first run."""

import numpy as np
import pytest

import workloads as wl
from oracle import micromag

torch = pytest.importorskip("torch")
import paper_2606_01114_gb300 as mm  # noqa: E402

pytestmark = pytest.mark.gpu

D = (2e-9, 2.5e-9, 3e-9)
TOL = {"f64": 1e-12, "ff": 1e-12, "f32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2606_01114_gb300 import build
    build.build()


def context(n, prec):
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32 if prec == "f32" else mm.MM_F64)
    mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.02, 0.0)
    if prec == "ff":
        mm.mm_set_fft_mode(ctx, mm.MM_FFT_FF)
    return ctx


def dev(a, prec):
    return torch.tensor(a, dtype=torch.float32 if prec == "f32" else torch.float64, device="cuda")


def rel(t, ref):
    return np.linalg.norm(t.double().cpu().numpy() - ref) / np.linalg.norm(ref)


# (nx, ny, nz): y padded to 16, 32, 40, ... 1024 and x likewise; the first and
# last side of a length's range; one block per plane up to nz = 8 (FP32) or 4
PLANE = [(2, 2, 1), (2, 3, 2), (17, 8, 4), (16, 9, 1), (33, 17, 2), (40, 21, 1), (41, 24, 4), (48, 25, 1), (49, 33, 8),
         (65, 40, 2), (81, 41, 1), (96, 48, 4), (97, 49, 1), (100, 25, 1), (129, 64, 2), (161, 81, 1), (193, 96, 8),
         (257, 97, 1), (321, 161, 2), (385, 193, 1), (7, 320, 1), (5, 321, 2), (3, 384, 1), (9, 511, 1), (511, 3, 1)]
# y, z and y as three kernels: nz above the plane kernel's, every z length
LINES = [(11, 7, 8), (5, 9, 16), (18, 20, 32), (6, 5, 64), (3, 7, 128), (7, 3, 256), (3, 3, 512), (6, 300, 16)]
# power-of-two meshes with long z lines: the z pass of the [c][z][y][kx]
# layout, every z length, a column tile that is not full, nx = 1 and ny = 1
ZCOLS = [(8, 4, 32), (64, 2, 32), (16, 8, 64), (4, 8, 128), (8, 4, 256), (2, 2, 512), (1, 4, 64), (64, 1, 32)]


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("n", PLANE + LINES + ZCOLS, ids=lambda n: "x".join(map(str, n)))
def test_demag_on_padded_lengths_matches_oracle(n, prec):
    p = micromag.Problem(n, D)
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, prec)
    md = dev(m, prec)
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, p.demag_fft(m)) < TOL[prec]
    mm.mm_destroy(ctx)


# FP64 meshes just above the size up to which a thread forms one output of a
# transform: the four-step of every x length, and of y on single layers
WIDE = [(16, 400, 16), (30, 320, 16), (33, 256, 16), (48, 256, 16), (64, 200, 8), (70, 160, 8), (90, 136, 8), (128, 100, 8),
        (150, 64, 16), (190, 64, 16), (256, 50, 8), (300, 40, 8), (350, 36, 8), (512, 25, 8), (200, 129, 1), (257, 81, 1)]


@pytest.mark.parametrize("n", WIDE, ids=lambda n: "x".join(map(str, n)))
def test_fp64_above_the_one_output_size_matches_oracle(n):
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, "f64")
    md = dev(m, "f64")
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, micromag.Problem(n, D).demag_fft(m)) < TOL["f64"]
    mm.mm_destroy(ctx)


@pytest.mark.parametrize("n", [(16, 8, 1), (32, 64, 2), (64, 32, 4), (8, 512, 1), (256, 16, 1), (512, 4, 2), (4, 4, 4)],
                         ids=lambda n: "x".join(map(str, n)))
def test_float_float_planes_match_oracle(n):
    p = micromag.Problem(n, D)
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, "ff")
    md = dev(m, "ff")
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, p.demag_fft(m)) < TOL["ff"]
    mm.mm_destroy(ctx)


# float-float z lines in registers (Pz = 16, 32, 64) and the Stockham pass
# beyond; column tiles that are not full, ny = 1
@pytest.mark.parametrize("n", [(16, 8, 8), (64, 4, 16), (8, 16, 32), (32, 1, 16), (4, 2, 64), (2, 4, 8)],
                         ids=lambda n: "x".join(map(str, n)))
def test_float_float_z_lines_match_oracle(n):
    m = wl.random_unit(n, seed=sum(n))
    ctx = context(n, "ff")
    md = dev(m, "ff")
    H = torch.full_like(md, float("nan"))
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, micromag.Problem(n, D).demag_fft(m)) < TOL["ff"]
    mm.mm_destroy(ctx)


@pytest.mark.parametrize("prec", ["f64", "ff", "f32"])
@pytest.mark.parametrize("n", [(32, 16, 2), (30, 21, 4), (19, 12, 16)], ids=lambda n: "x".join(map(str, n)))
def test_cell_wise_ms_and_the_unit_operator(n, prec):
    if prec == "ff" and any(v & (v - 1) for v in n):
        pytest.skip("float-float runs on power-of-two meshes")
    rng = np.random.default_rng(4)
    Ms = rng.uniform(4e5, 9e5, size=n[::-1])
    Ms[rng.random(Ms.shape) < 0.3] = 0.0
    m = wl.random_unit(n, seed=2)
    if prec == "f32":
        Ms = Ms.astype(np.float32).astype(np.float64)
    p = micromag.Problem(n, D, Ms_cell=Ms)
    ctx = context(n, prec)
    mm.mm_set_material_fields(ctx, Ms_cell=dev(Ms, prec))
    md = dev(m, prec)
    H = torch.empty_like(md)
    mm.mm_demag_field(ctx, md, H)
    assert rel(H, p.demag_fft(m)) < TOL[prec]
    # demag transpose: gm = Ms (-N g), the convolution with Ms = 1
    one = micromag.Problem(n, D, Ms=1.0)
    gm = torch.empty_like(md)
    mm.mm_demag_vjp(ctx, md, md, gm)
    assert rel(gm, Ms * one.demag_fft(m)) < TOL[prec]
    mm.mm_destroy(ctx)


def test_modes_of_the_other_passes_on_a_ragged_mesh():
    """The tensor-core y passes and the k-space product keep the 2n lengths
    and agree with the plane layout; switching back restores it."""
    n = (50, 256, 2)
    m = wl.random_unit(n, seed=9)
    ref = micromag.Problem(n, D).demag_fft(m)
    ctx = context(n, "f32")
    md = dev(m, "f32")
    H, H2 = torch.empty_like(md), torch.empty_like(md)
    mm.mm_demag_field(ctx, md, H)
    mm.mm_set_fft_mode(ctx, mm.MM_TC_TF32)
    mm.mm_demag_field(ctx, md, H2)
    assert rel(H2, ref) < TOL["f32"]
    mm.mm_set_fft_mode(ctx, 0)
    mm.mm_demag_field(ctx, md, H2)
    assert torch.equal(H, H2) and rel(H, ref) < TOL["f32"]
    mm.mm_destroy(ctx)
