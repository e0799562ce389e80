"""The fused update by independent warps (the library's choice of kernel for lattices of more
than 2^18 nodes): parity with the FP64 oracle
over the boundary modes at sizes that end strips, column pairs and row chunks everywhere, and
the same bits for a node wherever it lies in its strip and chunk.  (The small lattices of
test_parity_without_the_energy_equation run the tile kernel, which shares the lane's arithmetic;
test_sweep_modes_gpu.py has the sweep without the energy equation, checked by its name.)

Tolerance: the 1e-5 parity bound of the other update paths (test_parity_gpu.rel_errors); for
FP16 storage the bounds of the precision tests.
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


def lattice(nx, ny, p, **kw):
    from paper_1803_01756_gb300.lattice import KERNEL_FUSED, Lattice
    lat = Lattice(nx, ny, p, **kw)
    info = lat.info()
    assert (info["kernel"], info["cols_per_thread"]) == (KERNEL_FUSED, 2)
    assert info["tile_cols"] == (54 if p["thermal"] else 60)
    return lat


def compare(nx, ny, over, steps, storage=0):
    p = inputs.base_params(**{"u_amp": 0.03, "u_period": 50.0, **over})
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=nx + ny)
    lat = lattice(nx, ny, p, storage=storage)
    lat.write_fields(rho0)
    lat.step(steps)
    got = lat.read_fields()
    assert lat.status() == 0
    lat.close()
    o = oracle.Oracle(nx, ny, p)
    o.set_fields(rho0)
    o.step(steps)
    return rel_errors(got, o.fields())


SECTION_32 = dict(x_bc=0, u_amp=0.0, gy=-1e-4, T_wall_left=0.86, T_wall_right=0.80,
                  T_top_left=0.70, T_top_right=0.75, top_iso_x0=100, top_iso_x1=200,
                  bot_iso_x0=30, bot_iso_x1=280)


@pytest.mark.parametrize("nx,ny,over", [
    (521, 509, dict()),                      # odd width: the last column is alone in its pair
    (540, 487, dict(rho_w=1.0, tau_l=0.8)),  # ten whole strips
    (594, 443, dict(x_bc=2, p_amp_frac=0.1, u_period=60.0, gx=1e-4)),
    (515, 511, dict(x_bc=0)),                # periodic, odd: pairs lose their alignment
    (432, 611, dict(x_bc=0, y_bc=0)),
    (473, 557, dict(y_bc=0)),
    (502, 523, SECTION_32),
    (509, 521, dict(multiphase=0, gx=1e-5, rho_g=0.0)),
    (65537, 5, dict()),                      # fewer rows than the halo of a chunk
    (262145, 1, dict()),
    (5, 65537, dict(x_bc=0)),                # fewer columns than a strip
    (2, 131073, dict()),
])
def test_parity_above_the_two_pass_sizes(nx, ny, over):
    err = compare(nx, ny, over, 12)
    assert max(err.values()) <= TOL, err


@pytest.mark.parametrize("nx,ny,over", [
    (40, 21, dict()), (381, 34, dict(x_bc=0)), (61, 17, dict(y_bc=0)), (2, 9, dict()),
    (1, 7, dict(x_bc=0)), (9, 1, dict()), (5, 2, dict(x_bc=0, y_bc=0)), (60, 3, dict()),
    (120, 40, dict(x_bc=2, p_amp_frac=0.1)), (64, 33, dict(multiphase=0, gx=1e-5, rho_g=0.0)),
])
def test_parity_without_the_energy_equation(nx, ny, over):
    err = compare(nx, ny, dict(thermal=0, **over), 100)
    assert max(err.values()) <= TOL, err


def test_fp16_storage_against_the_oracle():
    err = compare(521, 509, dict(), 60, storage=2)
    assert err["rho"] <= 2e-3 and err["u"] <= 1.5e-2 and err["T"] <= 5e-4, err


@pytest.mark.parametrize("thermal", [1, 0])
@pytest.mark.parametrize("dx,dy", [(1, 0), (55, 0), (0, 1), (0, 7), (33, 200)])
def test_a_node_has_the_same_bits_wherever_it_lies(dx, dy, thermal):
    """In a periodic box the update commutes with a shift of the initial state: the shifted
    run holds every node in another column slot, strip, lane, row step and chunk."""
    nx, ny = 523, 504
    p = inputs.base_params(x_bc=0, y_bc=0, thermal=thermal)
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.05, seed=8)
    out = []
    for r in (rho0, np.roll(rho0, (dy, dx), (0, 1))):
        lat = lattice(nx, ny, p)
        lat.write_fields(r)
        lat.step(40)
        out.append(lat.read_fields())
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(np.roll(a, (dy, dx), (0, 1)), b)


@pytest.mark.parametrize("nx,ny", [(4096, 512), (1237, 531)])
def test_graph_replay_and_dependent_launch_give_the_bits_of_single_launches(nx, ny):
    """16-update graphs with dependent launches against one launch at a time with a
    synchronisation behind each."""
    import torch
    p = inputs.workload("channel_4096x512")["params"]
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=6)
    out = []
    for one in (False, True):
        lat = lattice(nx, ny, p)
        lat.set_graph(not one)
        lat.write_fields(rho0)
        for _ in range(83 if one else 1):
            lat.step(1 if one else 83)
            torch.cuda.synchronize()
        out.append(lat.read_fields())
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
