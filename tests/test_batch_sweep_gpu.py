"""A batch on the warp sweep: more lattices than one launch takes (48), uneven sizes down to a
few nodes, odd step counts and both parities of the graph chunks.  Lattices on the library's
kernel choice run the same arithmetic alone (tile kernel) and batched, so their fields are equal
bit for bit, with 16-bit storage too.
"""
import numpy as np
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [0, 2], ids=["f32", "f16"])
@pytest.mark.parametrize("n,x_bc", [(53, 1), (5, 0)])
def test_batch_equals_lattices_alone(n, x_bc, storage):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    from paper_1803_01756_gb300.lattice import Batch, Lattice
    u = inputs.uniform01(4 * n, 77).reshape(n, 4)
    specs = []
    for k in range(n):
        nx, ny = int(2 + u[k, 0] * 150), int(1 + u[k, 1] * 40)
        p = inputs.base_params(x_bc=x_bc, Gw=inputs.wall_strength_for_angle(45.0 + 90.0 * u[k, 2]),
                               u_period=float(200 + int(1800 * u[k, 3])))
        specs.append((nx, ny, p, inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, k)))

    def make():
        out = []
        for nx, ny, p, rho0 in specs:
            out.append(Lattice(nx, ny, p, storage=storage))
            out[-1].write_fields(rho0)
        return out

    alone, batched = make(), make()
    b = Batch(batched, graph=True)
    for steps in (19, 32, 2):
        b.step(steps)
        for lat in alone:
            lat.step(steps)
    for x, y in zip(alone, batched):
        assert x.t == y.t == 53
        for f, g in zip(x.read_fields(), y.read_fields()):
            assert np.array_equal(f, g)
    b.close()
    for lat in alone + batched:
        lat.close()
