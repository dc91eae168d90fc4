"""What a context promises beside its results: no allocation and no wait after
mm_init_mesh in the calls of the hot path, the octant of the 2n lengths on every
mesh, and no device memory beyond the arrays its passes use."""

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


# both sides ragged and above 32 (a chirp-z length each at 2n), one odd side,
# narrow sides, a power of two beside a ragged side, powers of two
@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 1e-5)])
@pytest.mark.parametrize("n", [(50, 37, 4), (9, 64, 2), (3, 5, 1), (48, 33, 16), (32, 16, 2)],
                         ids=lambda n: "x".join(map(str, n)))
def test_first_kspace_product_can_be_captured(n, prec, tol):
    """The product on the spectrum of a library transform is the demag field,
    and the first call on a context allocates nothing and does not wait: it is
    recorded into a graph."""
    dt = torch.float64 if prec == "f64" else torch.float32
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F64 if prec == "f64" else mm.MM_F32)
    mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.02, 0.0)
    m = wl.random_unit(n, seed=sum(n))
    pad = [2 * v if v > 1 else 1 for v in n]
    grid = torch.zeros(3, pad[2], pad[1], pad[0], dtype=dt, device="cuda")
    grid[:, :n[2], :n[1], :n[0]] = 8e5 * torch.tensor(m, dtype=dt, device="cuda")
    spec = torch.fft.rfftn(grid, dim=(1, 2, 3)).contiguous()
    work = torch.empty_like(spec)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    mm.mm_set_stream(ctx, stream)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        work.copy_(spec)
        mm.mm_kspace_product(ctx, work)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    H = torch.fft.irfftn(work, s=pad[::-1], dim=(1, 2, 3))[:, :n[2], :n[1], :n[0]]
    ref = micromag.Problem(n, D).demag_fft(m)
    assert np.linalg.norm(H.double().cpu().numpy() - ref) < tol * np.linalg.norm(ref)
    mm.mm_destroy(ctx)
