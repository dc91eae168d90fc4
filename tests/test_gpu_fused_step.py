"""The fused x inverse / cell / x forward kernel of small FP32 meshes against
the float64 oracle: the effective field, one RK4 step, one adaptive step and the
gradient of an RK4 step, at one, two and four cell rows per block with a last
block that is not full, at both kinds of x length, with vacuum, anisotropy and
DMI, and on a mesh just above the size up to which the kernel is taken.

Tolerances are the library's own for FP32 (1e-5 relative L2; 1e-4 for the
gradient), set before the first run."""

import numpy as np
import pytest

import workloads as wl
from oracle import micromag

torch = pytest.importorskip("torch")
import paper_2606_01114_gb300 as mm  # noqa: E402

pytestmark = pytest.mark.gpu

D = (2e-9, 2.5e-9, 3e-9)
# rows ny nz: below 304 (one a block), below 608 (two), four; x lengths 16 to 512
MESHES = [(100, 25, 1), (12, 19, 16), (33, 61, 8), (40, 303, 1), (70, 83, 8), (130, 333, 2), (500, 99, 2), (24, 500, 8),
          (300, 401, 1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2606_01114_gb300 import build
    build.build()


def rel(t, ref, on=1.0):
    return np.linalg.norm((t.double().cpu().numpy() - ref) * on) / np.linalg.norm(ref * on)


@pytest.mark.parametrize("vacuum", [False, True], ids=["uniform", "vacuum-dmi"])
@pytest.mark.parametrize("n", MESHES, ids=lambda n: "x".join(map(str, n)))
def test_field_and_steps_match_oracle(n, vacuum):
    m = wl.random_unit(n, seed=sum(n))
    Ms = None
    if vacuum:
        rng = np.random.default_rng(sum(n))
        Ms = rng.uniform(4e5, 9e5, size=n[::-1]).astype(np.float32).astype(np.float64)
        Ms[rng.random(Ms.shape) < 0.3] = 0.0
    kw = dict(A=1.3e-11, alpha=0.1, Ku=1e5, Ms_cell=Ms, D=1e-3 if vacuum else 0.0)
    p = micromag.Problem(n, D, **kw)
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32)
    mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.1, 1e5)
    if vacuum:
        mm.mm_set_material_fields(ctx, Ms_cell=torch.tensor(Ms, dtype=torch.float32, device="cuda"))
        mm.mm_set_dmi(ctx, 1e-3, mm.MM_DMI_INTERFACIAL)
    m0 = torch.tensor(m, dtype=torch.float32, device="cuda")
    H = torch.full_like(m0, float("nan"))
    mm.mm_effective_field(ctx, m0, H)
    assert rel(H, p.h_eff(m)) < 1e-5
    on = 1.0 if Ms is None else Ms > 0      # a vacuum cell keeps its m here and has none in the oracle
    md = m0.clone()
    mm.mm_rk4_trajectory(ctx, md, 1e-14, 2)
    assert rel(md, p.rk4_step(p.rk4_step(m, 1e-14), 1e-14), on) < 1e-5
    md = m0.clone()
    mm.mm_llg_step(ctx, md, 0.0, 2e-14, mm.MM_RKF45, 1.0)
    ref = micromag.rkf45_step(p, m, 0.0, 2e-14, 1.0)[0]
    assert rel(md, ref, on) < 1e-5
    if not vacuum:
        lam = torch.tensor(wl.random_unit(n, seed=7), dtype=torch.float32, device="cuda")
        # the trajectory's tape (fused kernels) and the single step's own recomputation
        a, b = lam.clone(), lam.clone()
        ga, gb = torch.zeros(ctx.shape1, device="cuda"), torch.zeros(ctx.shape1, device="cuda")
        mm.mm_rk4_trajectory_vjp(ctx, m0, 1e-14, 1, a, ga)
        mm.mm_rk4_step_vjp(ctx, m0, 1e-14, b, gb)
        assert float((a - b).norm() / b.norm()) < 1e-4
        assert float((ga - gb).norm() / gb.norm()) < 1e-4
    mm.mm_destroy(ctx)
