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
        p = inputs.base_params(**{"Gw": -1.2 + 0.02 * k, "u_amp": 0.03,
                                  "u_period": 60.0 + 7 * k, **over})
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
