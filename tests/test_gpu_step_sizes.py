"""The mixed tendency without tuning, on both sides of the sizes where the choice
of the element kernel changes (few z-lines per SM, a column per SM), against the
float64 one."""
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
