"""Wind diagnostics on warped layers on both sides of the size from which they run
in two launches: every node has its own reference density and lumped mass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from synth.vortex import random_state  # noqa: E402
from tests.test_gpu_remesh import LZ, background_rho  # noqa: E402


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("warp", [None, (500.0, 2, 3)])
@pytest.mark.parametrize("N,nz,nx,ny,half", [(4, 3, 16, 16, 70e3), (4, 3, 17, 17, 70e3), (2, 20, 45, 46, 20e3), (4, 97, 17, 16, 500e3),
                                              (4, 9, 36, 36, 60e3), (2, 3, 112, 112, 100e3), (2, 200, 65, 64, 20e3)])
def test_diag_levels_at_node_heights(sem, N, nz, nx, ny, half, warp):
    m = sem.sem_mesh_create(300e3, 300e3, LZ, nx, ny, nz, N, warp=warp)
    xyz = sem.sem_mesh_coords_host(m)
    q = random_state(xyz.T, LZ, 8)
    d = sem.sem_diag(m, sem.sem_params_default(), torch.from_numpy(np.ascontiguousarray(q)).cuda(), half)
    near = (np.abs(xyz[0]) <= half + 1e-6) & (np.abs(xyz[1]) <= half + 1e-6)
    s = np.sqrt(q[1] ** 2 + q[2] ** 2) / (background_rho(xyz[2]) + q[0])
    w = sem.sem_mesh_mass_host(m) * near
    num, den = (w * s).reshape(-1, m.NZ).sum(0), w.reshape(-1, m.NZ).sum(0)
    assert abs(d["max_wind"] / s[near].max() - 1) < 1e-12
    assert abs(d["max_mean_wind"] / (num / den).max() - 1) < 1e-12
