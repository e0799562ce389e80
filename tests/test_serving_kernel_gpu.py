"""The kernel of a served job: a job that leaves the kernel to the library has the bits of a
default lattice in every storage; one that names a kernel runs on the fused kernel, also where
it is large enough to be stepped alone."""
import ctypes

import numpy as np
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


def jobs():
    """(nx, ny, params, updates): small ones in two groups of modes, one stepped alone."""
    p = inputs.base_params(u_period=300.0)
    return [(200, 50, p, 40), (96, 33, dict(p, Gw=-1.15), 70), (600, 450, p, 25),
            (120, 40, dict(p, thermal=0), 33), (1024, 1024, p, 20)]


def serve(storage, kernel):
    """The jobs through lbm_submit with the kernel of their parameters, or through
    Server.submit (kernel None)."""
    from paper_1803_01756_gb300 import lattice as L
    srv = L.Server(hbm_budget=1 << 34, max_active=8, chunk_steps=16)
    ids = []
    for k, (nx, ny, p, steps) in enumerate(jobs()):
        rho0 = inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, k)
        if kernel is None:
            ids.append(srv.submit(nx, ny, p, steps, rho0, storage=storage))
            continue
        jid = ctypes.c_long()
        params = L.make_params(p, kernel=kernel, storage=storage)
        assert srv._lib.lbm_submit(srv._h, nx, ny, ctypes.byref(params), L._dptr(rho0), steps,
                                   ctypes.byref(jid)) == 0
        srv._shape[jid.value] = (ny, nx)
        ids.append(jid.value)
    out = []
    for j in ids:
        assert srv.wait(j, 300) == L.JOB_DONE
        out.append(srv.poll(j, fields=True)[1])
    srv.close()
    return out


def alone(storage, kernel):
    from paper_1803_01756_gb300.lattice import Lattice
    out = []
    for k, (nx, ny, p, steps) in enumerate(jobs()):
        lat = Lattice(nx, ny, p, kernel=kernel, storage=storage)
        lat.write_fields(inputs.noisy_density(nx, ny, inputs.RHO_V_086, 0.01, k))
        lat.step(steps)
        out.append(lat.read_fields())
        lat.close()
    return out


@pytest.mark.parametrize("storage,kernel", [(0, 0), (1, 0), (2, 0), (0, None)])
def test_library_choice_gives_the_bits_of_a_default_lattice(storage, kernel):
    for got, ref in zip(serve(storage, kernel), alone(storage, 0)):
        for a, b in zip(got, ref):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("storage,kernel", [(0, 2), (1, 2), (2, None), (1, None), (1, 5)])
def test_named_kernel_agrees_with_the_fused_kernel_alone(storage, kernel):
    """The FP32 parity bound of 1e-5; another kernel departs by 1e-3 and more in 16 bits."""
    for got, ref in zip(serve(storage, kernel), alone(storage, 2)):
        rho, ux, uy, T = got
        rr, rux, ruy, rT = ref
        assert np.abs(rho - rr).max() <= 1e-5 * np.abs(rr).max()
        assert np.hypot(ux - rux, uy - ruy).max() <= 1e-5 * max(np.hypot(rux, ruy).max(), 1e-3)
        assert np.abs(T - rT).max() <= 1e-5 * np.abs(rT).max()
