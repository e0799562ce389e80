"""Batches of more lattices than one launch of the warp sweep takes (48): several launches
beside one another, ordered with the caller's stream on both sides."""
import numpy as np
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def make(sizes, kernel=0):
    from paper_1803_01756_gb300.lattice import Lattice
    p = inputs.base_params(u_period=300.0)
    return [Lattice(nx, ny, p, kernel=kernel) for nx, ny in sizes]


def close(lats):
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("n", [48, 49, 97, 150])
def test_order_with_the_stream_of_the_caller(n, graph):
    """Fields written before, steps of two calls and fields read after, all enqueued on a side
    stream while it is still busy with other work."""
    import torch
    from paper_1803_01756_gb300.lattice import Batch
    sizes = [(30 + (7 * k) % 61, 5 + (5 * k) % 23) for k in range(n)]
    rho = [inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, k)
           for k, (nx, ny) in enumerate(sizes)]
    alone, batched = make(sizes), make(sizes)
    b = Batch(batched, graph=graph)
    s = torch.cuda.Stream()
    for lat, r in zip(batched, rho):
        lat.write_fields(r, stream=s)
    with torch.cuda.stream(s):
        busy = torch.randn(2048, 2048, device="cuda")
        for _ in range(20):
            busy = busy @ busy * 1e-2
    b.step(19, stream=s)
    b.step(16, stream=s)
    got = [lat.read_fields(stream=s) for lat in batched]
    for lat, r, g in zip(alone, rho, got):
        lat.write_fields(r)
        lat.step(35)
        for x, y in zip(lat.read_fields(), g):
            assert np.array_equal(x, y)
    b.close()
    close(alone + batched)


def test_launches_run_beside_one_another():
    """192 lattices in four launches against 48 in one, at the same tile height: the GPU is a
    tenth full with 48, so 192 take little longer (one launch after another: four times)."""
    import torch
    from paper_1803_01756_gb300.lattice import Batch

    def us(n):
        lats = make([(100, 32)] * n)
        b = Batch(lats, graph=True, tile_rows=16)
        b.step(32)
        best = 1e9
        for _ in range(5):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            b.step(64)
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1))
        b.close()
        close(lats)
        return best

    assert us(192) <= 2.5 * us(48)
