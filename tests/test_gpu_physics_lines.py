"""The mixed form's pass for the terms of the paper's runs in both equation
sets, at layer counts within, at and across its chunks, on 2:1 meshes: the total
within 1e-4 of the oracle and the added terms within 1e-3 of their own norm (the
bounds of the other physics tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import refstate, rhs as orhs  # noqa: E402
from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import dev, host, make_pair  # noqa: E402
from tests.test_gpu_physics import ADDED_TOL, PHYS  # noqa: E402

LEAVES = [(0, i, j) for i in range(3) for j in range(3) if (i, j) != (1, 1)] + [(1, 2 + a, 2 + b) for a in (0, 1) for b in (0, 1)]


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("eqset", ["C", "NC"])
@pytest.mark.parametrize("N,nz", [(2, 16), (2, 17), (3, 5), (3, 17), (4, 1), (4, 6), (4, 8), (4, 12), (4, 13), (5, 9), (6, 5)])
def test_terms_match_oracle(sem, N, nz, eqset):
    m, o, X, perm = make_pair(sem, L=300e3, Lz=12e3, nx=3, nz=nz, N=N, leaves=LEAVES)
    q_o = random_state(o.XG, o.Lz, 31, eqset)
    T_o = orhs.rhs(o, q_o, refstate.Params(**PHYS), eqset)
    D_o = T_o - orhs.rhs(o, q_o, refstate.Params(), eqset)
    q, out = dev(q_o[:, perm]), {}
    for name, phys in (("with", PHYS), ("without", {})):
        p = sem.sem_params_default(precision=sem.SEM_PREC_MIXED, eqset=int(eqset == "NC"), **phys)
        r = torch.full_like(q, float("nan"))
        sem.sem_rhs(m, p, q, r)
        out[name] = host(r)
    assert np.all(group_rel_l2(out["with"], T_o[:, perm]) <= 1e-4)
    added = out["with"] - out["without"]
    rows = [f for f in range(5) if np.linalg.norm(D_o[f]) > 1e-3 * np.linalg.norm(T_o[f])]
    for f in rows:   # fields whose added part stands out of the total's float32 rounding
        assert np.linalg.norm(added[f] - D_o[f][perm]) <= ADDED_TOL * np.linalg.norm(D_o[f]) + 2e-7 * np.linalg.norm(T_o[f])
    assert rows and sem.sem_status(m) == 0
