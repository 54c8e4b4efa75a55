"""The mixed tendency without tuning on meshes where the estimate that chooses the
element kernel's variant changes sides (chunks of a column against columns per SM),
against the float64 one, with and without the terms of the paper's runs."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import numpy as np  # noqa: E402

from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import host  # noqa: E402

LZ = 12e3
TERMS = dict(smag_cs=0.21, sponge_gamma=1.0, sponge_depth=4000.0)


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("terms", [False, True])
@pytest.mark.parametrize("eqset,N,nx,ny,nz", [
    (0, 2, 13, 13, 33), (0, 2, 26, 25, 33), (0, 3, 14, 14, 32), (0, 3, 25, 24, 32), (0, 4, 12, 12, 32), (0, 4, 30, 25, 32),
    (0, 4, 36, 36, 5), (0, 5, 12, 12, 17), (0, 5, 25, 24, 17), (0, 6, 12, 12, 14), (0, 6, 18, 17, 14),
    (1, 4, 12, 12, 28), (1, 4, 14, 14, 28), (1, 4, 25, 24, 17)])
def test_untuned_choice(sem, eqset, N, nx, ny, nz, terms):
    """Within 1e-4 (the mixed form's bound)."""
    m = sem.sem_mesh_create(nx * 75e3, ny * 75e3, LZ, nx, ny, nz, N)
    X = sem.sem_mesh_coords_host(m).T
    q = torch.from_numpy(np.ascontiguousarray(random_state(X, LZ, 6, "NC" if eqset else "C"))).cuda()
    out = []
    for prec in (sem.SEM_PREC_FP64, sem.SEM_PREC_MIXED):
        r = torch.full_like(q, float("nan"))
        sem.sem_rhs(m, sem.sem_params_default(eqset=eqset, precision=prec, **(TERMS if terms else {})), q, r)
        out.append(host(r))
    assert np.all(group_rel_l2(out[1], out[0]) <= 1e-4)
    assert sem.sem_status(m) == 0
