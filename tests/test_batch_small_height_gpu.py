"""Default tile height of the warp sweep for a few small lattices: short tiles, so that the SMs
get work (each tile sweeps 10 halo rows beside its own)."""
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nx,ny,rows", [(1, 1024, 128, 5), (12, 512, 64, 9), (48, 100, 32, 3),
                                          (24, 200, 50, 5), (1, 4096, 512, 22)])
def test_height_of_equal_lattices(n, nx, ny, rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("heights stated for 152 SMs")
    from paper_1803_01756_gb300 import build
    build.build()
    from paper_1803_01756_gb300.lattice import Batch, Lattice
    torch.cuda.set_device(0)
    lats = [Lattice(nx, ny, inputs.base_params()) for _ in range(n)]
    b = Batch(lats)
    assert b.info()["tile_rows"] == rows
    b.close()
    for lat in lats:
        lat.close()
