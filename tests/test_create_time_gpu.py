"""Preparation of a lattice does not grow with its height."""
import time

import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_tall_lattices_are_created_as_fast_as_wide_ones():
    """1 x 262144 nodes against 262144 x 1: 6.0 against 0.6 ms with an occupancy query for each of
    its 16,000 tile heights, 1.4 against 0.6 ms with one for each of the 10 heights of a tile
    (the rest is the memory of its 32-column pitch).  Bound: 3 ms apart, between the two."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    from paper_1803_01756_gb300.lattice import Lattice
    torch.cuda.set_device(0)
    p = inputs.base_params(x_bc=0)

    def ms(nx, ny):
        best = 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            lat = Lattice(nx, ny, p)
            best = min(best, 1e3 * (time.perf_counter() - t0))
            lat.close()
        return best

    tall, wide = ms(1, 1 << 18), ms(1 << 18, 1)
    print(f"\n1 x 262144: {tall:.2f} ms, 262144 x 1: {wide:.2f} ms")
    assert tall <= wide + 3.0
