"""Row chunks of the warp sweep: two CTAs per SM with taller chunks where a lattice is too small
for three (the halo's row steps are most of a short chunk), three where it is large."""
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,over,rows", [
    (1000, 300, dict(), 5), (1000, 300, dict(x_bc=0), 5), (520, 510, dict(), 6),
    (1237, 531, dict(), 7), (4096, 512, dict(), 22), (16384, 2048, dict(), 342),
    (1000, 300, dict(thermal=0), 4), (2048, 512, dict(), 12),
])
def test_chunk_height_follows_the_size(nx, ny, over, rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("heights stated for 152 SMs")
    from paper_1803_01756_gb300 import build
    build.build()
    from paper_1803_01756_gb300.lattice import Lattice
    torch.cuda.set_device(0)
    lat = Lattice(nx, ny, inputs.base_params(**over))
    assert lat.info()["tile_rows"] == rows
    lat.close()
