"""The warp sweep of a single lattice where other sizes run the tile kernel: without the energy
equation over the boundary modes, with each 16-bit storage, with liquid; and the status bits of
both kernels.  The kernel that ran is checked by its name in the per-launch timing.
Tolerance: the 1e-5 parity bound; for 16-bit storage the bounds of the precision tests.
"""
import numpy as np
import pytest

import oracle
from paper_1803_01756_gb300 import inputs
from test_parity_gpu import TOL, rel_errors
from test_precision_gpu import CHANNEL_BOUNDS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def lattice(nx, ny, p, kernel, **kw):
    """A fresh lattice, after a look at which kernel its twin runs."""
    from paper_1803_01756_gb300.lattice import Lattice
    with Lattice(nx, ny, p, **kw) as twin:
        twin.timing_enable(True)
        twin.step(1)
        assert set(twin.timing_get()) == {kernel}
    return Lattice(nx, ny, p, **kw)


def compare(nx, ny, over, steps, rho0=None, **kw):
    p = inputs.base_params(**{"u_amp": 0.03, "u_period": 50.0, **over})
    if rho0 is None:
        rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=nx + ny)
    with lattice(nx, ny, p, "k_sweep", **kw) as lat:
        lat.write_fields(rho0)
        lat.step(steps)
        got = lat.read_fields()
        assert lat.status() == 0
    o = oracle.Oracle(nx, ny, p)
    o.set_fields(rho0)
    o.step(steps)
    return rel_errors(got, o.fields())


NO_FORCE = dict(multiphase=0, gx=1e-5, rho_g=0.0)


@pytest.mark.parametrize("nx,ny,over", [
    (521, 509, dict()),                                    # odd width
    (540, 487, dict(tau_l=0.8, rho_w=1.0, gy=-1e-5, g_omega=0.01)),  # nine whole strips
    (541, 485, dict(x_bc=2, p_amp_frac=0.1, u_period=60.0, gx=1e-4)),
    (515, 511, dict(x_bc=0)), (432, 611, dict(x_bc=0, y_bc=0)), (473, 557, dict(y_bc=0)),
    (509, 521, NO_FORCE), (515, 511, dict(x_bc=0, **NO_FORCE)),
    (513, 512, dict(x_bc=0, y_bc=0, **NO_FORCE)), (473, 557, dict(y_bc=0, **NO_FORCE)),
    (131073, 2, dict()), (2, 131073, dict()), (262145, 1, dict()), (121, 2168, dict(x_bc=0)),
])
def test_parity_without_the_energy_equation(nx, ny, over):
    err = compare(nx, ny, dict(over, thermal=0), 12)
    assert max(err.values()) <= TOL, err


@pytest.mark.parametrize("storage", [1, 2], ids=["bf16", "f16"])
@pytest.mark.parametrize("nx,ny,over", [
    (521, 509, dict()), (515, 511, dict(x_bc=0)), (432, 611, dict(x_bc=0, y_bc=0)),
    (594, 443, dict(x_bc=2, p_amp_frac=0.1, u_period=60.0, gx=1e-4)),
    (509, 521, NO_FORCE), (473, 557, dict(thermal=0)), (53, 5000, dict()),
])
def test_16bit_storage_against_the_oracle(nx, ny, over, storage):
    err = compare(nx, ny, over, 24, storage=storage)
    bound = CHANNEL_BOUNDS[{1: "bf16", 2: "f16"}[storage]]
    assert all(err[k] <= bound[k] for k in bound), err


def test_parity_with_liquid():
    """Drops on strip and chunk borders: the whole range of the equation of state."""
    nx, ny = 620, 430
    y, x = np.mgrid[0:ny, 0:nx].astype(float)
    r = np.min([np.hypot(x - a, y - b) for a, b in ((54, 12), (268, 200), (610, 429))], axis=0)
    rho0 = inputs.RHO_V_086 + (inputs.RHO_L_086 - inputs.RHO_V_086) * 0.5 * (
        1 - np.tanh((r - 8) / 2))
    err = compare(nx, ny, dict(x_bc=0, u_amp=0.0), 12, rho0)
    assert max(err.values()) <= TOL, err


# States outside the model's domain on a node and its neighbours (the update streams before it
# computes the density), and the status bit of each (lbm.h).
def poison(kind, rho, T, at, p, Tc):
    ny, nx = rho.shape
    rows = [y for y in range(at[0] - 1, at[0] + 2) if 0 <= y < ny]
    patch = np.ix_(rows, [x % nx for x in range(at[1] - 1, at[1] + 2)])
    if kind == "nan":
        rho[patch] = np.nan
    elif kind == "psi":  # P > rho / 3: a hot vapour
        T[patch] = 0.6
    elif kind == "rho":
        rho[patch] = -0.01
    elif kind == "pole":
        rho[patch] = 1.001 / p["eos_b"]
    else:
        T[patch] = -1e-3 * Tc


BITS = {"nan": 1, "psi": 2, "rho": 4, "pole": 8, "T": 16}


@pytest.mark.parametrize("kind", sorted(BITS))
@pytest.mark.parametrize("nx,ny,kernel", [(521, 509, "k_sweep"), (157, 61, "k_tile")])
@pytest.mark.parametrize("where", ["corner", "inside", "last column"])
def test_status_bits(nx, ny, kernel, kind, where):
    p = inputs.base_params(x_bc=0)
    rho = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=3)
    at = {"corner": (0, 0), "inside": (ny // 2, 54), "last column": (ny - 1, nx - 1)}[where]
    with lattice(nx, ny, p, kernel) as lat:
        T = np.full((ny, nx), 0.86 * lat.Tc)
        lat.write_fields(rho, T)
        lat.step(3)
        assert lat.status() == 0
        poison(kind, rho, T, at, p, lat.Tc)
        lat.write_fields(rho, T)
        lat.step(1)
        assert lat.status(clear=True) & BITS[kind]
        assert lat.status() == 0


@pytest.mark.parametrize("nx,ny,kernel", [(521, 509, "k_sweep"), (157, 61, "k_tile")])
def test_unstable_parameters_are_reported(nx, ny, kernel):
    """Conductivity beyond the stability bound of the energy update."""
    from paper_1803_01756_gb300.lattice import LbmError
    p = inputs.base_params(x_bc=0, **{"lambda": 40.0})
    with lattice(nx, ny, p, kernel) as lat:
        lat.write_fields(inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, seed=2))
        lat.step(400)
        with pytest.raises(LbmError) as ei:
            lat.read_fields()
        assert ei.value.code == -4 and lat.status() != 0
