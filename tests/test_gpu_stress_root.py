"""The eddy viscosity's square root is correctly rounded in the paper's set.

In a pure shear u = +-g y on boxes with sides of powers of two the stress's
invariant is the square of g exactly, so with a g of at most 12 bits the
viscosity (C_s delta)^2 g and every flux ahead of the weights are exact.  The
same fluxes follow from a shear of a power of two with C_s times g, whose root is
exact in any arithmetic; nothing else moves u, so both tendencies have the same
bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


def tendency(sem, m, y, g, cs):
    q = torch.zeros((5, m.NG), dtype=torch.float64, device="cuda")
    q[1] = g * y.abs()   # kinks on element faces: zero and the domain's edge
    p = sem.sem_params_default(precision=sem.SEM_PREC_MIXED, eqset=sem.SEM_EQ_NONCONSERVATIVE, smag_cs=cs, f=0.0)
    out = torch.empty_like(q)
    return sem.sem_rhs(m, p, q, out)[1].clone()


@pytest.mark.parametrize("nz", [1, 2])
def test_root_of_a_square_is_exact(sem, nz):
    h = 65536.0
    m = sem.sem_mesh_create(4 * h, 4 * h, 8192.0, 4, 4, nz, 2)
    y = torch.from_numpy(sem.sem_mesh_coords_host(m)[1].copy()).cuda()
    for g in np.random.default_rng(0).integers(2049, 4096, 100).tolist():
        one = tendency(sem, m, y, g * 2.0 ** -24, 0.25)
        two = tendency(sem, m, y, 2.0 ** -12, 0.25 * g * 2.0 ** -12)
        assert float(one.abs().max()) > 0
        assert torch.equal(one, two), g
