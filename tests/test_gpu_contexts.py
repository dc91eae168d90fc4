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
# narrow sides, a power of two beside a ragged side, powers of two with and
# without a side below the shortest padded length
@pytest.mark.parametrize("prec,tol", [("f64", 1e-12), ("f32", 1e-5)])
@pytest.mark.parametrize("n", [(50, 37, 4), (9, 64, 2), (3, 5, 1), (48, 33, 16), (32, 16, 2), (2, 2, 1), (2, 16, 4), (16, 2, 1)],
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


# a plain context of the plane layout holds its state arrays (11 vector fields,
# Ms, A), the octant of the 2n lengths, and the planes, octant and line buffer
# of its passes; not the arrays of passes it does not run
@pytest.mark.parametrize("n", [(512, 512, 4), (256, 256, 4)], ids=lambda n: "x".join(map(str, n)))
def test_device_memory_of_a_plain_context(n):
    nx, ny, nz = n
    N, P, K, Hs = nx * ny * nz, 2 * ny, nx + 1, (nx + 16) // 16 * 16
    octants = 6 * (nz + 1) * (ny + 1) * Hs + K * 6 * (nz + 1) * ((P // 2 + 4) // 4 * 4)
    want = 4 * (35 * N + octants + 2 * K * 3 * nz * ny)
    warm = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32)      # the library's own modules and streams
    mm.mm_destroy(warm)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F32)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    mm.mm_destroy(ctx)
    assert want < used < want + 20 * 2 ** 21      # allocations come in granules of 2 MB


def test_modes_after_a_plain_context_allocate_what_they_need():
    """Power-of-two meshes of the plane layout: the tensor-core mode and the
    float-float mode of a mesh too large for its plane kernel run the passes
    whose arrays a plain context does not hold; switching back restores it."""
    for n, prec, mode, tol in (((64, 256, 2), "f32", mm.MM_TC_TF32, 1e-5), ((32, 256, 4), "f64", mm.MM_FFT_FF, 1e-12)):
        m = wl.random_unit(n, seed=2)
        ref = micromag.Problem(n, D).demag_fft(m)
        ctx = mm.mm_init_mesh(*n, *D, precision=mm.MM_F64 if prec == "f64" else mm.MM_F32)
        mm.mm_set_material(ctx, 8e5, 1.3e-11, 0.02, 0.0)
        md = torch.tensor(m, dtype=torch.float64 if prec == "f64" else torch.float32, device="cuda")
        H = torch.empty_like(md)
        for k in (mode, 0, mode):
            mm.mm_set_fft_mode(ctx, k)
            mm.mm_demag_field(ctx, md, H)
            assert np.linalg.norm(H.double().cpu().numpy() - ref) < tol * np.linalg.norm(ref)
        mm.mm_destroy(ctx)
