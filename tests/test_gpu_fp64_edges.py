"""The float64 form's reciprocal and pressure series at the edges of their ranges."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import refstate, rhs as orhs  # noqa: E402
from synth.vortex import random_state  # noqa: E402
from tests.helpers import group_rel_l2  # noqa: E402
from tests.test_gpu_parity import dev, host, make_pair  # noqa: E402


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


@pytest.mark.parametrize("eqset,warp", [("C", None), ("NC", None), ("C", (500.0, 1, 2))])
def test_reciprocal_scales_with_the_density(sem, eqset, warp):
    """p00 and the state times 2^k: every product, sum and power-of-two
    quotient of the tendency scales exactly.  Within the reciprocal's own range
    the bits are equal; beyond 2^+-100 it is the division, correctly rounded,
    and a reciprocal may differ by its last bit there (once in some hundreds:
    the third-order step leaves 2^-63 before its rounding): 1e-14 of the norm
    is 45 such units in every term.  Two densities are not finite."""
    m, o, X, perm = make_pair(sem, L=300e3, Lz=12e3, nx=3, nz=5, N=4, warp=warp)
    rng = np.random.default_rng(5)
    q0 = random_state(o.XG, o.Lz, 7, eqset)[:, perm]
    # a second density beside the reference's: below zero, in the paper's set (whose
    # pressure needs rho theta > 0) above it
    q0[0] = (-2.5 if eqset == "C" else 1.5) * rng.integers(0, 2, m.NG) + rng.uniform(-0.01, 0.01, m.NG)
    scaled = np.array([1, 1, 1, 1, 1] if eqset == "C" else [1, 0, 0, 0, 0])

    def tendency(k, q):
        f = np.where(scaled[:, None], 2.0 ** k, 1.0)
        p = sem.sem_params_default(eqset=int(eqset == "NC"), p00=1e5 * 2.0 ** k)
        out = torch.empty((5, m.NG), dtype=torch.float64, device="cuda")
        return host(sem.sem_rhs(m, p, dev(q * f), out)) / f

    base = tendency(0, q0)
    assert np.all(np.isfinite(base))
    for k in (-90, -1, 50, 95):
        np.testing.assert_array_equal(tendency(k, q0), base)
    for k in (-150, -101, -100, -99, -98, 98, 99, 100, 101, 102, 150):
        assert np.all(group_rel_l2(tendency(k, q0), base) <= 1e-14), k
    for bad in (np.inf, np.nan):
        q = q0.copy()
        q[0, m.NG // 3] = bad
        np.testing.assert_array_equal(np.isfinite(tendency(0, q)), np.isfinite(tendency(150, q)))


@pytest.mark.parametrize("R_d", [287.0, 700.0, 920.0, 974.0])
@pytest.mark.parametrize("eqset", ["C", "NC"])
def test_pressure_of_any_gas(sem, R_d, eqset):
    """The float64 tendency within its 1e-12 of the oracle for ratios of
    specific heats from 1.4 to 33, pressures on both sides of where the series
    ends."""
    prm = refstate.Params(R_d=R_d)
    m, o, X, perm = make_pair(sem, L=300e3, Lz=12e3, nx=3, nz=3, N=3)
    q_o = random_state(o.XG, o.Lz, 3, eqset)
    ref = refstate.reference_state(o.XG[:, 2], prm)
    x = np.random.default_rng(1).choice([-0.035, -0.0312, 0.01, 0.0312, 0.0313], o.NG)
    # rho theta' = x (rho theta)0
    q_o[4] = x * ref["rhotheta0"] if eqset == "C" else (x * ref["rhotheta0"] - q_o[0] * ref["theta0"]) / (ref["rho0"] + q_o[0])
    want = orhs.rhs(o, q_o, prm, eqset)
    out = torch.empty((5, m.NG), dtype=torch.float64, device="cuda")
    sem.sem_rhs(m, sem.sem_params_default(R_d=R_d, eqset=int(eqset == "NC")), dev(q_o[:, perm]), out)
    assert np.all(group_rel_l2(host(out), want[:, perm]) <= 1e-12)
