"""The float64 form's chunked element kernel against the oracle where a column
spans several layer chunks of every order (the level carried between chunks, a
last chunk of one layer), on 2:1 meshes, with pressures on both sides of the
series' range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import refstate, rhs as orhs  # noqa: E402
from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import dev, host, make_pair  # noqa: E402

PRM = refstate.Params()
LEAVES = [(0, i, j) for i in range(3) for j in range(3) if (i, j) != (1, 1)] + [(1, 2 + a, 2 + b) for a in (0, 1) for b in (0, 1)]


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("N,nz", [(2, 16), (2, 33), (3, 8), (3, 9), (4, 8), (4, 9), (4, 17), (5, 4), (5, 9), (6, 2),
                                  (6, 5), (4, 1)])
def test_chunked_tendency_matches_oracle(sem, N, nz):
    m, o, X, perm = make_pair(sem, L=300e3, Lz=12e3, nx=3, nz=nz, N=N, leaves=LEAVES)
    q_o = random_state(o.XG, o.Lz, 21)
    far = q_o.copy()
    rng = np.random.default_rng(0)
    far[4] = refstate.reference_state(o.XG[:, 2], PRM)["rhotheta0"] * rng.uniform(-0.3, 0.3, size=o.NG) * (
        rng.random(o.NG) < 0.5)
    for state in (q_o, far):
        T_o = orhs.rhs(o, state, PRM)
        out = torch.full((5, m.NG), float("nan"), dtype=torch.float64, device="cuda")
        sem.sem_rhs(m, sem.sem_params_default(), dev(state[:, perm]), out)
        assert np.all(group_rel_l2(host(out), T_o[:, perm]) <= 1e-12)
    assert sem.sem_status(m) == 0
