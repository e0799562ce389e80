"""The tile kernel, the library's choice on lattices of at most 2^18 nodes, over the cases of the
parity and precision tests: boundary modes, degenerate sizes, liquid, 16-bit storage, graph
replay; and the two passes of LBM_KERNEL_TWOPASS where they are named.  The tolerances are those
of the tests that the cases come from.
"""
import numpy as np
import pytest

import oracle
from paper_1803_01756_gb300 import inputs
from test_parity_gpu import CASES, TOL, rel_errors
from test_precision_gpu import (CHANNEL_BOUNDS, LONG_BOUNDS, RADIUS_BOUNDS, STORAGES,  # noqa: F401
                                channel_reference, contact_angle, drop_reference,
                                equimolar_radius, errors, long_reference, sessile_drop)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def kernels_of(nx, ny, p, **kw):
    """The kernels of an update, by the names of the per-launch timing."""
    from paper_1803_01756_gb300.lattice import Lattice
    with Lattice(nx, ny, p, **kw) as lat:
        lat.timing_enable(True)
        lat.step(1)
        return set(lat.timing_get())


def run(nx, ny, p, rho0, steps, **kw):
    from paper_1803_01756_gb300.lattice import Lattice
    assert kernels_of(nx, ny, p, **kw) == {"k_tile"}
    with Lattice(nx, ny, p, **kw) as lat:
        lat.write_fields(rho0)
        lat.step(steps)
        assert lat.status() == 0
        return lat.read_fields()


def parity(nx, ny, p, rho0, steps):
    o = oracle.Oracle(nx, ny, p)
    o.set_fields(rho0)
    o.step(steps)
    err = rel_errors(run(nx, ny, p, rho0, steps), o.fields())
    assert max(err.values()) <= TOL, err


def liquid(nx, ny, drops, radius):
    y, x = np.mgrid[0:ny, 0:nx].astype(float)
    r = np.min([np.hypot(x - a, y - b) for a, b in drops], axis=0)
    return inputs.RHO_V_086 + (inputs.RHO_L_086 - inputs.RHO_V_086) * 0.5 * (
        1 - np.tanh((r - radius) / 2))


@pytest.mark.parametrize("over", [dict(), dict(thermal=0)])
@pytest.mark.parametrize("nx,ny", [(200, 50), (521, 509)])
def test_a_named_path_runs_as_named(nx, ny, over):
    """At most 2^18 nodes and more: the two passes are two launches (one without the energy
    equation)."""
    from paper_1803_01756_gb300.lattice import KERNEL_TWOPASS
    names = kernels_of(nx, ny, inputs.base_params(**over), kernel=KERNEL_TWOPASS)
    assert names == ({"k_stream_collide"} if over else {"k_stream_collide", "k_energy_rk4"})


@pytest.mark.parametrize("nx,ny,over", CASES)
def test_parity_over_the_boundary_modes(nx, ny, over):
    p = inputs.base_params(**{"u_amp": 0.03, "u_period": 50.0, **over})
    parity(nx, ny, p, inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=nx * 1000 + ny), 200)


@pytest.mark.parametrize("nx,ny,over", [(2, 9, dict()), (1, 7, dict(x_bc=0)), (9, 1, dict()),
                                        (5, 2, dict(y_bc=0, x_bc=0)), (64, 3, dict())])
def test_parity_of_degenerate_sizes(nx, ny, over):
    parity(nx, ny, inputs.base_params(**over),
           inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=11), 30)


@pytest.mark.parametrize("nx,ny,drops,radius,over,steps", [
    (48, 32, [(24.0, -0.5)], 10, dict(x_bc=0, u_amp=0.0), 300),
    (420, 40, [(150.0, 12.0), (290.0, 27.0)], 8, dict(u_amp=0.02, u_period=400.0), 100),
])
def test_parity_with_liquid(nx, ny, drops, radius, over, steps):
    parity(nx, ny, inputs.base_params(**over), liquid(nx, ny, drops, radius), steps)


@pytest.mark.parametrize("name,steps", [("channel_200x50", 1000), ("condensation_100x300", 300)])
def test_parity_of_the_workloads(name, steps):
    w = inputs.workload(name)
    parity(w["nx"], w["ny"], w["params"], inputs.initial_density(w), steps)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_channel_error_against_oracle(storage, channel_reference):  # noqa: F811
    w = inputs.workload("channel_200x50")
    got = run(w["nx"], w["ny"], w["params"], inputs.initial_density(w), 1000,
              storage=STORAGES[storage])
    err = errors(got, channel_reference)
    assert all(err[k] <= b for k, b in CHANNEL_BOUNDS[storage].items()), err


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_liquid_drop_density_and_contact_angle(storage, drop_reference):  # noqa: F811
    p, rho_ref, ca_ref = drop_reference
    rho = run(80, 40, p, sessile_drop(), 4000, storage=STORAGES[storage])[0]
    assert np.abs(rho - rho_ref).max() / rho_ref.max() <= {"f32": 2e-4, "f16": 8e-2,
                                                           "bf16": 0.25}[storage]
    assert abs(contact_angle(rho) - ca_ref) <= {"f32": 0.01, "f16": 0.5, "bf16": 6.0}[storage]
    assert abs(equimolar_radius(rho) - equimolar_radius(rho_ref)) <= RADIUS_BOUNDS[storage]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_benchmark_channel_20000_updates(storage, long_reference):  # noqa: F811
    p, rho0, ref = long_reference
    err = errors(run(128, 32, p, rho0, 20000, storage=STORAGES[storage]), ref)
    assert all(err[k] <= b for k, b in LONG_BOUNDS[storage].items()), err


@pytest.mark.parametrize("over", [dict(), dict(thermal=0), dict(x_bc=2, p_amp_frac=0.1,
                                                                u_period=60.0)])
def test_graph_replay_equals_one_launch_per_update(over):
    from paper_1803_01756_gb300.lattice import Lattice
    nx, ny = 150, 40
    p = inputs.base_params(**{"u_amp": 0.03, "u_period": 50.0, **over})
    rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=21)
    out = []
    for graph in (True, False):
        with Lattice(nx, ny, p) as lat:
            lat.set_graph(graph)
            lat.write_fields(rho0)
            for n in (5, 40):
                lat.step(n)
            lat.timing_enable(True)
            lat.step(17)
            lat.timing_enable(False)
            for n in (37, 32):
                lat.step(n)
            assert lat.t == 131
            out.append(lat.read_fields())
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_checkpoint_resume_is_bitwise():
    from paper_1803_01756_gb300.lattice import Lattice
    w = inputs.workload("channel_200x50")
    with Lattice(w["nx"], w["ny"], w["params"]) as a, Lattice(w["nx"], w["ny"], w["params"]) as b:
        a.write_fields(inputs.initial_density(w))
        a.step(70)
        b.write_state(a.read_state())
        a.step(30)
        b.step(30)
        assert b.t == 100
        for x, y in zip(a.read_fields(), b.read_fields()):
            assert np.array_equal(x, y)
