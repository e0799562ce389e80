"""LBM_FUSED_TILE and LBM_FUSED_CPT act on lattices of the library's kernel choice too."""
import pytest

from paper_1803_01756_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_01756_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def ran(nx, ny, over):
    from paper_1803_01756_gb300.lattice import Lattice
    with Lattice(nx, ny, inputs.base_params(**over)) as lat:
        lat.timing_enable(True)
        lat.step(1)
        i = lat.info()
        return set(lat.timing_get()), (i["tile_cols"], i["tile_rows"], i["cols_per_thread"])


@pytest.mark.parametrize("nx,ny,over", [(521, 509, dict()), (200, 50, dict(thermal=0))])
def test_variables_set_the_cta_sweep(nx, ny, over, monkeypatch):
    assert "k_fused_step" not in ran(nx, ny, over)[0]
    monkeypatch.setenv("LBM_FUSED_TILE", "60,7")
    assert ran(nx, ny, over) == ({"k_fused_step"}, (60, 7, 1))
    monkeypatch.delenv("LBM_FUSED_TILE")
    monkeypatch.setenv("LBM_FUSED_CPT", "2")
    names, (_, _, cpt) = ran(nx, ny, over)
    assert names == {"k_fused_step"} and cpt == 2


def test_small_lattices_with_the_energy_equation_keep_their_kernel(monkeypatch):
    monkeypatch.setenv("LBM_FUSED_TILE", "60,7")
    assert ran(200, 50, dict())[0] == {"k_tile"}
