"""A batch of lattices on the library's kernel choice gives the bits of the same lattices alone,
in every mode of the physics and every storage: the tile kernel and the warp sweep alone, the
batched warp sweep together.
"""
import numpy as np
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu

NO_FORCE = dict(multiphase=0, rho_g=0.0, gx=1e-5)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    torch.cuda.set_device(0)


# one lattice above 2^18 nodes (the warp sweep alone), the others at the edges of strips of 54
# and 60 columns, of row chunks and of CTAs of four warps
SIZES = [(521, 509), (241, 33), (54, 16), (61, 7), (107, 1), (2, 90), (300, 40)]


def make(over, storage=0, sizes=SIZES, kernels=None):
    from paper_1803_01756_gb300.lattice import Lattice
    out = []
    for k, (nx, ny) in enumerate(sizes):
        p = inputs.base_params(**{"Gw": -1.2 + 0.02 * (k % 7), "u_amp": 0.03,
                                  "u_period": 60.0 + 7 * (k % 7), **over})
        out.append(Lattice(nx, ny, p, storage=storage, kernel=kernels[k] if kernels else 0))
        out[-1].write_fields(inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, k))
    return out


def same_bits(alone, batched):
    for x, y in zip(alone, batched):
        assert x.t == y.t
        for f, g in zip(x.read_fields(), y.read_fields()):
            assert np.array_equal(f, g), (x.nx, x.ny)


def close(*lats):
    for group in lats:
        for lat in group:
            lat.close()


@pytest.mark.parametrize("storage", [0, 1, 2], ids=["f32", "bf16", "f16"])
@pytest.mark.parametrize("over", [
    dict(), dict(thermal=0), NO_FORCE, dict(thermal=0, **NO_FORCE),
    dict(thermal=0, x_bc=0), dict(x_bc=0, y_bc=0), dict(y_bc=0, thermal=0),
    dict(x_bc=2, p_amp_frac=0.1, gx=1e-4, **{"tau_l": 0.8}),
], ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "full")
def test_batch_gives_the_bits_of_the_lattices_alone(over, storage):
    from paper_1803_01756_gb300.lattice import Batch
    alone, batched = make(over, storage), make(over, storage)
    b = Batch(batched, graph=True)
    for steps in (17, 6):
        b.step(steps)
        for lat in alone:
            lat.step(steps)
    same_bits(alone, batched)
    b.close()
    close(alone, batched)


def rel_errors(got, ref):
    rho, ux, uy, T = got
    rr, rux, ruy, rT = ref
    return (np.abs(rho - rr).max() / np.abs(rr).max(),
            np.hypot(ux - rux, uy - ruy).max() / max(np.hypot(rux, ruy).max(), 1e-3),
            np.abs(T - rT).max() / np.abs(rT).max())


@pytest.mark.parametrize("storage", [0, 1, 2], ids=["f32", "bf16", "f16"])
@pytest.mark.parametrize("tiling", [(7, 94, 1), (40, 120, 2), (16, 244, 2)])
def test_a_tiling_does_not_change_the_results(tiling, storage):
    from paper_1803_01756_gb300.lattice import Batch
    alone, batched = make({}, storage), make({}, storage)
    b = Batch(batched)
    b.step(5)
    b.set_tiling(*tiling)
    assert b.info()["tile_rows"] == tiling[0]
    b.step(18)
    for lat in alone:
        lat.step(23)
    same_bits(alone, batched)
    b.close()
    close(alone, batched)


@pytest.mark.parametrize("tiling", [None, (24, 94, 1)])
@pytest.mark.parametrize("storage", [0, 2], ids=["f32", "f16"])
@pytest.mark.parametrize("n", [7, 53])
def test_each_lattice_of_a_mixed_batch_runs_its_own_kernel(n, storage, tiling):
    """Lattices of the library's choice beside ones of the named kernels.  The former keep the
    bits they have alone; the work-list kernel and the single-lattice kernels of the named paths
    compute the same update, so with 16-bit storage too those agree within the FP32 bound of
    1e-5 (a departure at the storage's precision is 1e-3 and more)."""
    from paper_1803_01756_gb300.lattice import Batch
    sizes = (SIZES[1:] + [(90 + 3 * k, 12 + k) for k in range(n)])[:n]
    kernels = [(0, 2, 0, 3, 0, 2, 5)[k % 7] for k in range(n)]
    over = dict(thermal=1)
    alone, batched = make(over, storage, sizes, kernels), make(over, storage, sizes, kernels)
    b = Batch(batched, graph=True)
    if tiling:
        b.set_tiling(*tiling)
        i = b.info()
        assert (i["tile_rows"], i["tile_cols"], i["cols_per_thread"]) == tiling
    for steps in (19, 32, 2):
        b.step(steps)
        for lat in alone:
            lat.step(steps)
    for k, (x, y) in enumerate(zip(alone, batched)):
        if kernels[k] != 0:
            assert max(rel_errors(y.read_fields(), x.read_fields())) <= 1e-5, k
        else:
            same_bits([x], [y])
    b.close()
    close(alone, batched)
