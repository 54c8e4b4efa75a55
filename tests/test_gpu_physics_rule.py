"""The mixed form's pass for the terms of the paper's runs on both sides of the
sizes where its kernel changes (thin meshes of orders 2 and 3 in the paper's set, a
column per SM at order 4 in the conservative one), against the float64 form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import host  # noqa: E402
from tests.test_gpu_physics import ADDED_TOL, PHYS  # noqa: E402

LZ = 12e3


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("eqset,N,n,nz", [(1, 2, 4, 1), (1, 2, 20, 2), (1, 2, 22, 2), (1, 2, 37, 7), (1, 2, 39, 7), (1, 2, 39, 8),
                                          (1, 3, 4, 1), (1, 3, 14, 2), (0, 4, 12, 12), (0, 4, 13, 12),
                                          (0, 4, 4, 17), (0, 4, 4, 25), (0, 4, 13, 25)])
def test_terms_by_either_kernel(sem, eqset, N, n, nz):
    """The total within 1e-4, the added terms within ADDED_TOL of their own norm
    (the bounds of the other physics tests)."""
    m = sem.sem_mesh_create(30e3 * n, 30e3 * n, LZ, n, n, nz, N)
    X = sem.sem_mesh_coords_host(m).T
    q = torch.from_numpy(np.ascontiguousarray(random_state(X, LZ, 31, "NC" if eqset else "C"))).cuda()
    out = {}
    for prec in (sem.SEM_PREC_FP64, sem.SEM_PREC_MIXED):
        for phys in (PHYS, {}):
            r = torch.full_like(q, float("nan"))
            sem.sem_rhs(m, sem.sem_params_default(precision=prec, eqset=eqset, **phys), q, r)
            out[prec, bool(phys)] = host(r)
    T, mixed = out[sem.SEM_PREC_FP64, True], out[sem.SEM_PREC_MIXED, True]
    assert np.all(group_rel_l2(mixed, T) <= 1e-4)
    D, added = T - out[sem.SEM_PREC_FP64, False], mixed - out[sem.SEM_PREC_MIXED, False]
    rows = [f for f in range(5) if np.linalg.norm(D[f]) > 1e-3 * np.linalg.norm(T[f])]
    for f in rows:
        assert np.linalg.norm(added[f] - D[f]) <= ADDED_TOL * np.linalg.norm(D[f]) + 2e-7 * np.linalg.norm(T[f])
    assert rows and sem.sem_status(m) == 0
