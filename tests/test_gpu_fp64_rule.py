"""The float64 tendency on both sides of every size where its element kernel
changes (layers by order and columns per SM), against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import refstate, rhs as orhs  # noqa: E402
from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import dev, host, make_pair  # noqa: E402

PRM = refstate.Params()


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("N,n,nz", [(2, 3, 1), (2, 3, 2), (2, 22, 3), (2, 22, 4), (3, 12, 1), (3, 12, 2), (3, 13, 2),
                                    (3, 13, 3), (3, 22, 3), (3, 22, 4), (4, 3, 3), (4, 3, 4), (4, 13, 9), (5, 12, 6),
                                    (5, 13, 5), (5, 13, 6), (5, 13, 9), (6, 3, 1), (6, 13, 3)])
def test_tendency_by_either_kernel(sem, N, n, nz):
    m, o, X, perm = make_pair(sem, L=75e3 * n, Lz=12e3, nx=n, nz=nz, N=N)
    q_o = random_state(o.XG, o.Lz, 17)
    out = torch.full((5, m.NG), float("nan"), dtype=torch.float64, device="cuda")
    sem.sem_rhs(m, sem.sem_params_default(), dev(q_o[:, perm]), out)
    assert np.all(group_rel_l2(host(out), orhs.rhs(o, q_o, PRM)[:, perm]) <= 1e-12)
    assert sem.sem_status(m) == 0
