"""Default tile height of a batch on the warp sweep: a height between the listed ones where it
makes one wave, and the bits of the lattices alone at it."""
import numpy as np
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mix", [(16, 77), (20, 21)])
def test_heights_between_the_listed_ones(n, mix):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    from paper_1803_01756_gb300.lattice import Batch, Lattice
    u = inputs.uniform01(4 * n, mix).reshape(n, 4)
    sizes = [(int(256 + v[0] * 1792), int(32 + v[1] * 224)) for v in u]
    p = inputs.base_params(u_amp=0.02, u_period=2000.0)

    def make():
        out = []
        for k, (nx, ny) in enumerate(sizes):
            out.append(Lattice(nx, ny, p))
            out[-1].write_fields(inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, k))
        return out

    alone, batched = make(), make()
    b = Batch(batched)
    info = b.info()
    assert info["tile_rows"] % 4 == 0 and info["tile_rows"] >= 24
    # one wave: four warps a CTA, strips of 54 columns in groups of four
    rows = info["tile_rows"]
    ctas = sum(-(-(-(-(nx + 1) // 54)) // 4) * -(-ny // rows) for nx, ny in sizes)
    assert 4 * ctas <= info["grid"]
    b.step(7)
    for x, y in zip(alone, batched):
        x.step(7)
        for f, g in zip(x.read_fields(), y.read_fields()):
            assert np.array_equal(f, g)
    b.close()
    for lat in alone + batched:
        lat.close()
