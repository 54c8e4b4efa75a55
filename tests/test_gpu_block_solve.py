"""The block solver of the transfer with four right-hand sides per CTA, which it
takes once its blocks give every SM one: a last group with one right-hand side
left, and systems that end at different passes (a field of zeros, one of a much
smaller size, one whose values span many decades)."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import adapt, mesh as om, transfer as otr  # noqa: E402
from synth.vortex import random_state  # noqa: E402
from tests.helpers import node_perm  # noqa: E402

LZ = 12e3


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


def blocks(sem, m):
    """Number of coupled blocks and size of the largest: nodes that the
    hanging rows with several weights link."""
    hmap, hh, hw = sem.sem_mesh_hmap_host(m)
    hh = hh[(hw != 0).sum(1) >= 2]
    a = sp.coo_matrix((np.ones(hh.size), (hh.ravel(), np.repeat(hh[:, :1], hh.shape[1]).ravel())), shape=(m.NH, m.NH))
    lab = sp.csgraph.connected_components(a, directed=False)[1][np.unique(hh)]
    return len(np.unique(lab)), np.bincount(lab).max()


@pytest.mark.parametrize("N,nz,left", [(4, 32, 1), (3, 33, 0), (5, 26, 3)])
def test_four_right_hand_sides(sem, N, nz, left):
    m = sem.sem_mesh_create(400e3, 400e3, LZ, 8, 8, nz, N, lvl_max=3)
    o = om.OracleMesh(400e3, 400e3, LZ, 8, 8, nz, N)
    perm = node_perm(sem.sem_mesh_coords_host(m), o.XG)
    q_o = random_state(o.XG, LZ, 9)
    rng = np.random.default_rng(1)
    q_o[1] *= 10.0 ** rng.uniform(-12, 2, q_o.shape[1])
    q_o[3] = 0.0
    q_o[4] *= 1e-90
    refine = {(0, 1, 1), (0, 5, 5), (0, 5, 6), (0, 1, 6)}
    fl = np.repeat(np.array([tuple(l) in refine for l in sem.sem_mesh_leaves_host(m).tolist()], dtype=np.int8), nz)
    fl_o = np.repeat(np.array([tuple(l) in refine for l in o.leaves], dtype=np.int8), nz)
    new = sem.sem_transfer_plan(m, fl)
    n_blocks, largest = blocks(sem, new)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n_blocks * 5 * new.NZ >= 4 * sms and 128 * largest <= 200 * 1024   # the solver's rule
    assert 5 * new.NZ % 4 == left
    new_o, org = adapt.update_leaves(o.leaves, fl_o, nz, 8, 8, 3)
    o2, want = otr.transfer(o, new_o, org, q_o)
    want = want[:, node_perm(sem.sem_mesh_coords_host(new), o2.XG)]
    got = torch.full((5, new.NG), float("nan"), dtype=torch.float64, device="cuda")
    sem.sem_transfer(m, new, torch.from_numpy(np.ascontiguousarray(q_o[:, perm])).cuda(), got)
    got = got.cpu().numpy()
    assert np.all(got[3] == 0.0) and sem.sem_status(new) == 0
    for f in (0, 1, 2, 4):
        assert np.linalg.norm(got[f] - want[f]) <= 1e-12 * np.linalg.norm(want[f])
