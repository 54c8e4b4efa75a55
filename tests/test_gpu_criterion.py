"""The speed criterion's own kernel against the general one, bit for bit.

A criterion slot beyond the thresholds in use that names another variable sends
the call to the general kernel, which evaluates every node in float64 with the
same rounded operations; element maxima and flags have to be equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.test_gpu_remesh import make, states  # noqa: E402

THR = [5.0, 10.0, 15.0]


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


def both(sem, m, q, **params):
    out = []
    for last in (sem.SEM_CRIT_SPEED, sem.SEM_CRIT_VORTICITY):
        p = sem.sem_params_default(lvl_max=3, criterion=[0] * (sem.SEM_MAX_THRESHOLDS - 1) + [last], **params)
        flags = torch.full((m.Ne,), 9, dtype=torch.int8, device="cuda")
        cmax = torch.full((m.Ne,), -1.0, dtype=torch.float64, device="cuda")
        sem.sem_adapt_flags(m, p, torch.from_numpy(np.ascontiguousarray(q)).cuda(), flags, cmax)
        out.append((flags.cpu().numpy(), cmax.cpu().numpy()))
    return out


@pytest.mark.parametrize("warp", [None, (500.0, 2, 3)])
@pytest.mark.parametrize("eqset", [0, 1])
@pytest.mark.parametrize("N,nz", [(2, 3), (2, 130), (3, 1), (3, 90), (4, 16), (4, 63), (4, 64), (5, 7), (6, 43)])
def test_speed_kernel_equals_general_kernel(sem, N, nz, eqset, warp):
    m = make(sem, N, nz, warp=warp)
    for name, q in states(sem, m, eqset):
        (f1, c1), (f2, c2) = both(sem, m, q, eqset=eqset, thresholds=THR)
        np.testing.assert_array_equal(c1, c2, err_msg=name)
        np.testing.assert_array_equal(f1, f2, err_msg=name)


@pytest.mark.parametrize("N,nz,n", [(2, 1, 54), (2, 2, 28), (2, 3, 4), (3, 1, 40), (3, 2, 28), (3, 3, 13), (4, 1, 28),
                                    (4, 2, 20), (4, 3, 13), (5, 1, 22), (5, 2, 16), (6, 1, 18), (6, 2, 14), (6, 3, 13)])
def test_thin_meshes(sem, N, nz, n):
    """One to three layers where the speed kernel takes over from the general one."""
    m = make(sem, N, nz, n)
    for name, q in states(sem, m, 0):
        (f1, c1), (f2, c2) = both(sem, m, q, thresholds=THR)
        np.testing.assert_array_equal(c1, c2, err_msg=name)
        np.testing.assert_array_equal(f1, f2, err_msg=name)


def test_density_whose_inverse_square_underflows(sem):
    """1 / rho^2 below float32's normal range: the float32 bounds lose bits there."""
    m = make(sem, 4, 4)
    rng = np.random.default_rng(0)
    z = sem.sem_mesh_coords_host(m)[2]
    rho = 8e24 * 1.16e-5 * np.exp(-z / 9e3)   # about the reference density
    q = np.zeros((5, m.NG))
    q[0] = rho * rng.uniform(0.3, 0.9, m.NG)
    q[1] = (rho + q[0]) * 0.09 * (1.0 + 4e-5 * rng.uniform(-1, 1, m.NG))
    (f1, c1), (f2, c2) = both(sem, m, q, p00=8e24, thresholds=[0.01, 0.05, 0.08])
    assert 0.05 < c2.min() and c2.max() < 0.2
    np.testing.assert_array_equal(c1, c2)
    np.testing.assert_array_equal(f1, f2)
