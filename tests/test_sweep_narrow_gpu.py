"""The warp sweep on lattices of one, two and three strips, above 2^18 nodes: every warp of a
CTA has a tile, and the fields keep to the 1e-5 parity bound of the other update paths.
"""
import pytest

import oracle
from paper_1803_01756_gb300 import inputs
from test_parity_gpu import TOL, rel_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def ran(lat):
    """The kernels of an update, by the names of the per-launch timing."""
    lat.timing_enable(True)
    lat.step(1)
    names = set(lat.timing_get())
    lat.timing_enable(False)
    return names


@pytest.mark.parametrize("nx,strips", [(53, 1), (54, 2), (107, 2), (108, 3)])
def test_row_chunks_of_a_narrow_lattice_fill_the_warps(nx, strips):
    """One wave of three CTAs of four warps an SM: as many row chunks as it has warps for."""
    import torch
    from paper_1803_01756_gb300.lattice import Lattice
    ny = (1 << 20) // strips
    lat = Lattice(nx, ny, inputs.base_params())
    assert ran(lat) == {"k_sweep"}
    warps = 12 * torch.cuda.get_device_properties(0).multi_processor_count
    assert lat.info()["tile_rows"] <= -(-ny // (warps // (strips if strips < 3 else 4)))
    lat.close()


@pytest.mark.parametrize("nx,ny,over", [
    (53, 5000, dict()), (40, 6563, dict(x_bc=0)), (107, 2461, dict()), (64, 4099, dict(y_bc=0)),
    (96, 2733, dict(x_bc=0, y_bc=0)), (108, 2431, dict()), (161, 1637, dict(x_bc=0)),
    (60, 4371, dict(thermal=0)), (7, 37453, dict(x_bc=2, p_amp_frac=0.1)),
])
def test_parity_of_narrow_lattices(nx, ny, over):
    from paper_1803_01756_gb300.lattice import Lattice
    p = inputs.base_params(**{"u_amp": 0.03, "u_period": 50.0, **over})
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=nx + ny)
    lat = Lattice(nx, ny, p)
    assert ran(lat) == {"k_sweep"}
    lat.close()
    lat = Lattice(nx, ny, p)
    lat.write_fields(rho0)
    lat.step(12)
    got = lat.read_fields()
    assert lat.status() == 0
    lat.close()
    o = oracle.Oracle(nx, ny, p)
    o.set_fields(rho0)
    o.step(12)
    err = rel_errors(got, o.fields())
    assert max(err.values()) <= TOL, err
