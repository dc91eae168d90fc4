"""Contexts of different meshes used from different host threads at once: one
kernel serves both with different amounts of shared memory, and neither thread
may take the other's away.  Calls on one context do not overlap; each context
has its own stream.  The results are those of the same run alone, bit for bit
(the RK4 path has no atomics)."""

import threading

import pytest

import workloads as wl

torch = pytest.importorskip("torch")
import paper_2606_01114_gb300 as mm  # noqa: E402

pytestmark = pytest.mark.gpu

D = (2e-9, 2.5e-9, 3e-9)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2606_01114_gb300 import build
    build.build()


# the plane kernel of two heights, the fused cell kernel of one and four rows a
# block, the FP64 z pass of two lengths, the float-float plane of two lengths
PAIRS = [("f32", (100, 250, 8), (100, 250, 4)), ("f32", (300, 100, 1), (300, 70, 8)), ("f64", (64, 64, 16), (64, 64, 32)),
         ("f64", (20, 300, 1), (20, 500, 1))]


@pytest.mark.parametrize("prec,na,nb", PAIRS)
def test_threads_with_contexts_of_different_meshes(prec, na, nb):
    dt = torch.float32 if prec == "f32" else torch.float64
    meshes = (na, nb)
    streams = [torch.cuda.Stream() for _ in meshes]
    ctxs = [mm.mm_init_mesh(*n, *D, precision=mm.MM_F32 if prec == "f32" else mm.MM_F64, stream=s)
            for n, s in zip(meshes, streams)]
    m0 = [torch.tensor(wl.random_unit(n, seed=3), dtype=dt, device="cuda") for n in meshes]
    alone = [m.clone() for m in m0]
    out = [[m.clone() for _ in range(4)] for m in m0]
    torch.cuda.synchronize()
    for c, m in zip(ctxs, alone):
        mm.mm_rk4_trajectory(c, m, 1e-14, 100)
    failed = []
    gate = threading.Barrier(len(meshes))

    def work(k):
        try:
            gate.wait()
            for m in out[k]:
                mm.mm_rk4_trajectory(ctxs[k], m, 1e-14, 100)
        except Exception as e:      # noqa: BLE001 - reported below, in the main thread
            failed.append((meshes[k], str(e)))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(meshes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    torch.cuda.synchronize()
    for a, runs in zip(alone, out):
        for m in runs:
            assert torch.equal(a, m)
    for c in ctxs:
        mm.mm_destroy(c)
