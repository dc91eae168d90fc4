"""mm_relax against the same adaptive run taken step by step.

A batch of mm_relax reuses the demag field of its torque check as the first
trial's first stage, and stops when the end time has been reached; mm_llg_step
does neither.  Both run the same kernels on the same values in the same order
(the largest error is the only reduction, and a maximum does not depend on
order), so states, times and step counts are equal."""

import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
import paper_2606_01114_gb300 as mm  # noqa: E402

pytestmark = pytest.mark.gpu

D = (2e-9, 2.5e-9, 3e-9)
STEPS = 27
# fused stage, four kernels a stage, the [c][z][y][kx] passes; float-float in
# both layouts
RUNS = [("f32", (64, 64, 4)), ("f32", (33, 61, 8)), ("f32", (200, 200, 4)), ("f32", (32, 16, 16)), ("f64", (50, 40, 2)),
        ("f64", (16, 16, 16)), ("ff", (64, 32, 2)), ("ff", (16, 16, 8))]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2606_01114_gb300 import build
    build.build()


def context(n, prec, vacuum):
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32 if prec == "f32" else mm.MM_F64)
    mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.5, 1e5)
    dt = torch.float32 if prec == "f32" else torch.float64
    if prec == "ff":
        mm.mm_set_fft_mode(ctx, mm.MM_FFT_FF)
    if vacuum:
        rng = np.random.default_rng(sum(n))
        Ms = rng.uniform(4e5, 9e5, size=n[::-1])
        Ms[rng.random(Ms.shape) < 0.2] = 0.0
        mm.mm_set_material_fields(ctx, Ms_cell=torch.tensor(Ms, dtype=dt, device="cuda"))
    return ctx, torch.tensor(wl.random_unit(n, seed=sum(n)), dtype=dt, device="cuda")


def step_by_step(ctx, m, t_max, max_steps):
    """(times, step lengths, rejected trials) of the run mm_relax makes."""
    t, dt, times, lengths, rejected = 0.0, min(1e-14, t_max), [0.0], [], 0
    while t < t_max and len(lengths) < max_steps:
        dt = min(dt, t_max - t)
        t, dt, _ = mm.mm_llg_step(ctx, m, t, dt, mm.MM_RKF45, 1e-5)
        rejected += mm.mm_step_stats(ctx)[1]
        lengths.append(t - times[-1])
        times.append(t)
    return times, lengths, rejected


@pytest.mark.parametrize("vacuum", [False, True], ids=["uniform", "vacuum"])
@pytest.mark.parametrize("prec,n", RUNS, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
def test_relax_is_the_same_run(prec, n, vacuum):
    ctx, m0 = context(n, prec, vacuum)
    a = m0.clone()
    times, lengths, rejected = step_by_step(ctx, a, float("inf"), STEPS)
    # three batches and a part of one, ended by the number of steps
    b = m0.clone()
    with pytest.raises(mm.MMError):
        mm.mm_relax(ctx, b, 1.0, 0.0, STEPS)
    assert mm.mm_step_stats(ctx)[:3] == (STEPS, rejected, times[-1])
    assert torch.equal(a, b)
    # ended by the time: inside the first batch, and inside a later one
    for k in (3, 16):
        t_max = times[k] + 0.4 * lengths[k]
        a, b = m0.clone(), m0.clone()
        end = step_by_step(ctx, a, t_max, 1000)
        t, steps = mm.mm_relax(ctx, b, t_max, 0.0, 1000)
        assert (t, steps) == (end[0][-1], len(end[1])) and mm.mm_step_stats(ctx)[1] == end[2]
        assert torch.equal(a, b)
    mm.mm_destroy(ctx)


def test_relax_after_a_rejected_first_trial():
    """A batch whose first trial is rejected evaluates the field of the same
    state again; the run still is the same."""
    n = (64, 64, 4)
    ctx, m0 = context(n, "f32", False)
    mm.mm_set_material(ctx, 8e5, 1.3e-9, 0.5, 1e5)      # a hundred times stiffer: the first 1e-14 s are too long
    a, b = m0.clone(), m0.clone()
    times, _, rejected = step_by_step(ctx, a, float("inf"), 12)
    assert rejected > 0
    with pytest.raises(mm.MMError):
        mm.mm_relax(ctx, b, 1.0, 0.0, 12)
    assert mm.mm_step_stats(ctx)[:3] == (12, rejected, times[-1]) and torch.equal(a, b)
    mm.mm_destroy(ctx)
