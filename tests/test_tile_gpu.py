"""The tile kernel (the library's choice on lattices of at most 2^18 nodes):
parity with the FP64 oracle where a CTA sweeps several tiles and at the largest size, and the
same bits for a node wherever it lies.  The boundary modes, degenerate sizes,
16-bit storage and graph replay are in test_tile_modes_gpu.py.
Tolerance: the 1e-5 parity bound of the other update paths.
"""
import numpy as np
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


@pytest.mark.parametrize("nx,ny,over", [
    (512, 512, dict()),
    (53, 4001, dict(x_bc=0)),
    (107, 2003, dict(y_bc=0)),
    (1601, 47, dict(x_bc=2, p_amp_frac=0.1, u_period=60.0, gx=1e-4)),
    (701, 301, dict(x_bc=0, u_amp=0.0, gy=-1e-4, T_wall_left=0.86, T_wall_right=0.80,
                    T_top_left=0.70, T_top_right=0.75, top_iso_x0=100, top_iso_x1=200,
                    bot_iso_x0=30, bot_iso_x1=280)),
    (131072, 2, dict()),
    (600, 400, dict(thermal=0, x_bc=0)),
])
def test_parity_with_several_tiles_per_block(nx, ny, over):
    from paper_1803_01756_gb300.lattice import Lattice
    p = inputs.base_params(**{"u_amp": 0.03, "u_period": 50.0, **over})
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=nx + ny)
    lat = Lattice(nx, ny, p)
    assert lat.info()["cols_per_thread"] == 2
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


@pytest.mark.parametrize("thermal", [1, 0])
@pytest.mark.parametrize("dx,dy", [(1, 0), (55, 0), (0, 1), (0, 9), (33, 20)])
def test_a_node_has_the_same_bits_wherever_it_lies(dx, dy, thermal):
    """In a periodic box the update commutes with a shift of the initial state: the shifted
    run holds every node in another column slot, strip, lane, warp and tile."""
    from paper_1803_01756_gb300.lattice import Lattice
    nx, ny = 331, 253
    p = inputs.base_params(x_bc=0, y_bc=0, thermal=thermal)
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.05, seed=8)
    out = []
    for r in (rho0, np.roll(rho0, (dy, dx), (0, 1))):
        lat = Lattice(nx, ny, p)
        lat.write_fields(r)
        lat.step(40)
        out.append(lat.read_fields())
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(np.roll(a, (dy, dx), (0, 1)), b)
