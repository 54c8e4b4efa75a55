"""The mixed form without tuning.

The mixed step on meshes on both sides of the size from which the column
residual and the two mirrors no longer fit L2 (the gather's loads and stores are
marked differently there), box and warped, against the float64 step; and the
tendency on both sides of the sizes where the choice of the element kernel
changes (few z-lines per SM, a column per SM), against the float64 one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import host  # noqa: E402

LZ = 12e3


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("warp", [None, (500.0, 2, 3)])
@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (17, 13, 3), (41, 39, 14), (47, 44, 16)])
def test_mixed_step_matches_float64(sem, nx, ny, nz, warp):
    """The increment of the step within 1e-4 (the mixed form's bound)."""
    m = sem.sem_mesh_create(nx * 75e3, ny * 75e3, LZ, nx, ny, nz, 4, warp=warp)
    q0 = torch.from_numpy(np.ascontiguousarray(random_state(sem.sem_mesh_coords_host(m).T, LZ, 5))).cuda()
    ref, w1, w2 = q0.clone(), torch.empty_like(q0), torch.empty_like(q0)
    sem.sem_step(m, sem.sem_params_default(), ref, w1, w2, 0.25)
    q, q32 = q0.clone(), torch.empty(q0.shape, dtype=torch.float32, device="cuda")
    work = torch.empty((10, m.NG), dtype=torch.float32, device="cuda")
    sem.sem_mirror(m, q, q32)
    sem.sem_step_mixed(m, sem.sem_params_default(precision=sem.SEM_PREC_MIXED), q, q32, work, 0.25)
    assert np.all(group_rel_l2(host(q - q0), host(ref - q0)) <= 1e-4)
    assert torch.equal(q32, sem.sem_mirror(m, q, torch.empty_like(q32)))
    assert sem.sem_status(m) == 0


@pytest.mark.parametrize("eqset", [0, 1])
@pytest.mark.parametrize("N,nx,ny,nz", [(2, 14, 11, 17), (3, 9, 8, 9), (3, 20, 15, 17), (3, 30, 21, 17), (4, 9, 8, 9),
                                        (4, 14, 11, 12), (4, 18, 14, 17), (4, 30, 21, 6), (5, 14, 11, 9),
                                        (6, 15, 10, 9), (6, 20, 15, 9)])
def test_untuned_tendency_matches_float64(sem, N, nx, ny, nz, eqset):
    """Within 1e-4 (the mixed form's bound)."""
    m = sem.sem_mesh_create(nx * 75e3, ny * 75e3, LZ, nx, ny, nz, N)
    X = sem.sem_mesh_coords_host(m).T
    q = torch.from_numpy(np.ascontiguousarray(random_state(X, LZ, 6, "NC" if eqset else "C"))).cuda()
    out = []
    for prec in (sem.SEM_PREC_FP64, sem.SEM_PREC_MIXED):
        r = torch.full_like(q, float("nan"))
        sem.sem_rhs(m, sem.sem_params_default(eqset=eqset, precision=prec), q, r)
        out.append(host(r))
    assert np.all(group_rel_l2(out[1], out[0]) <= 1e-4)
    assert sem.sem_status(m) == 0
