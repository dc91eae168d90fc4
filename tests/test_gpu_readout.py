"""Read-outs of a state: energies of a state that is not finite, and the
largest torque, which FP32 contexts filter in single precision and evaluate in
double where it can be the maximum.

The torque's tolerance: the reference is evaluated in double from the
library's own single-precision exchange and demag fields, which the torque
kernel forms by the same formulas, so the two can differ by the rounding of
the exchange terms (at most 32 units of 2^-24 of the largest term sum) and of
the anisotropy."""

import numpy as np
import pytest

import workloads as wl
from oracle import micromag

torch = pytest.importorskip("torch")
import paper_2606_01114_gb300 as mm  # noqa: E402

pytestmark = pytest.mark.gpu

D = (2e-9, 2.5e-9, 3e-9)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2606_01114_gb300 import build
    build.build()


def context(n, prec, **kw):
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32 if prec == "f32" else mm.MM_F64)
    mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.02, kw.get("Ku", 0.0))
    return ctx


def dev(a, prec):
    return torch.tensor(a, dtype=torch.float32 if prec == "f32" else torch.float64, device="cuda")


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("Ku,h", [(0.0, 0.0), (1e5, 0.0), (0.0, 1e4), (1e5, 1e4)])
def test_energies_of_a_state_that_is_not_finite(prec, value, Ku, h):
    n = (20, 13, 2)
    m = wl.random_unit(n, seed=1)
    m[0, 1, 7, 11] = value
    with np.errstate(all="ignore"):
        ref = micromag.Problem(n, D, Ku=Ku, h_ext=(0.0, h, 0.0)).energies(m)
    ctx = context(n, prec, Ku=Ku)
    mm.mm_set_external_field(ctx, 0.0, h, 0.0)
    E = np.array(mm.mm_energy(ctx, dev(m, prec)))
    # (the oracle's fifth term sums over the DMI field of every cell; without DMI the library reports zero)
    assert np.isnan(ref[:4]).all() and np.isnan(E[:4]).all() and E[4] == 0.0
    mm.mm_destroy(ctx)


def unit(a):
    return a / np.linalg.norm(a, axis=0, keepdims=True)


STATES = {
    "random": lambda n, r: unit(r.standard_normal((3, n[2], n[1], n[0]))),
    # near alignment along z, one cell tilted a little more than the rest: the
    # largest torque is a small difference of large fields
    "aligned": lambda n, r: unit(np.array([0.0, 0.0, 1.0])[:, None, None, None] + 1e-4 * r.standard_normal((3, n[2], n[1], n[0]))),
    # uniform: every torque is rounding and stray field
    "uniform": lambda n, r: unit(np.ones((3, n[2], n[1], n[0]))),
}


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("state", list(STATES))
@pytest.mark.parametrize("n", [(1, 1, 1), (7, 5, 1), (100, 25, 1), (64, 64, 4), (130, 90, 8)],
                         ids=lambda n: "x".join(map(str, n)))
def test_largest_torque_is_the_largest_over_all_cells(n, state, prec):
    rng = np.random.default_rng(sum(n))
    m = STATES[state](n, rng)
    Ms = rng.uniform(4e5, 9e5, size=n[::-1])
    if Ms.size > 1:
        Ms[rng.random(Ms.shape) < 0.3] = 0.0
    Ms.flat[0] = 5e5
    ctx = context(n, prec, Ku=2e5)
    Msd, md = dev(Ms, prec), dev(m, prec)
    mm.mm_set_material_fields(ctx, Ms_cell=Msd)
    H = torch.empty_like(md)
    mm.mm_exchange_field(ctx, md, H)
    hx = H.double().cpu().numpy()
    mm.mm_demag_field(ctx, md, H)
    hd = H.double().cpu().numpy()
    md64, Ms64 = md.double().cpu().numpy(), Msd.double().cpu().numpy()
    mag = Ms64 > 0
    inv = np.where(mag, 1.0 / np.where(mag, Ms64, 1.0), 0.0)
    ha = np.zeros_like(hx)
    ha[2] = 2 * 2e5 / micromag.MU0 * inv * md64[2]
    t = np.linalg.norm(np.cross(md64, hx + hd + ha, axis=0), axis=0) * inv
    # terms of the exchange sum: six bonds of at most 2 |m| each
    bond = sum(2 * 1.3e-11 / (micromag.MU0 * d * d) for d in D)
    scale = (2 * 2 * bond * inv + np.abs(hd).sum(0) + np.abs(ha).sum(0)) * np.abs(md64).sum(0) * inv
    eps = 2.0 ** -24 if prec == "f32" else 2.0 ** -53
    assert abs(mm.mm_max_torque(ctx, md) - t.max()) <= 32 * eps * scale.max()
    mm.mm_destroy(ctx)


def test_exchange_with_cell_wise_a_streams():
    """512x512x16 FP32 with Ms and A per cell: eight arrays (134 MB) at no less
    than 1.5 TB/s (1.6 before all bonds were loaded together, then 1.3)."""
    n = (512, 512, 16)
    ctx = context(n, "f32")
    g = torch.Generator(device="cuda").manual_seed(1)
    Ms = 4e5 + 5e5 * torch.rand(ctx.shape1, generator=g, device="cuda")
    mm.mm_set_material_fields(ctx, Ms_cell=Ms, A_cell=2e-17 * Ms)
    m = torch.randn(ctx.shape3, generator=g, device="cuda")
    H = torch.empty_like(m)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(9):
        a.record()
        for _ in range(10):
            mm.mm_exchange_field(ctx, m, H)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) / 10 * 1e-3)
    assert 8 * 4 * Ms.numel() / sorted(times)[4] > 1.5e12
    mm.mm_destroy(ctx)
