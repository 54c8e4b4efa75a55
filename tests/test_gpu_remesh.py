"""The kernels between the steps at the sizes where they can go wrong: the
speed criterion (bounded in float32, decided in float64) bit for bit, the wind
diagnostics, the network's features and the solution transfer, for every order,
on 2:1 meshes, with layer counts around the kernels' chunks and with states of
zeros, ties, values outside float32's range, NaN and non-positive densities."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import adapt, mlp as omlp, transfer as otr  # noqa: E402
from oracle import mesh as om  # noqa: E402
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


def two_level(n):
    """Leaves of an n x n base with column (1, 1) refined."""
    out = [(0, i, j) for i in range(n) for j in range(n) if (i, j) != (1, 1)]
    return out + [(1, 2 + a, 2 + b) for a in (0, 1) for b in (0, 1)]


def make(sem, N, nz, n=4, leaves=None, warp=None):
    return sem.sem_mesh_create(300e3, 300e3, LZ, n, n, nz, N, leaves=leaves or two_level(n), lvl_max=3, warp=warp)


def local_lines(sem, m, q):
    """q [5, NG] on every column line, [5, Ncol, Nq, NZ]; hanging lines summed in
    order with a rounded product and a rounded addition per term."""
    hmap, hh, hw = sem.sem_mesh_hmap_host(m)
    q = q.reshape(5, m.NH, m.NZ)
    hang = np.zeros((5, max(len(hh), 1), m.NZ))
    for i in range(m.N + 1 if len(hh) else 0):
        hang = hang + hw[None, :, i, None] * q[:, hh[:, i]]
    out = np.where(hmap[None, :, :, None] >= 0, q[:, np.maximum(hmap, 0)], hang[:, np.maximum(-1 - hmap, 0)])
    return out


def background_rho(z, g=9.81, th=300.0, N=0.01, R=287.0, cp=1004.0, p00=1e5):
    pi = 1.0 + g * g / (cp * th * N * N) * (np.exp(-N * N * z / g) - 1.0)
    return p00 * pi ** ((cp - R) / R) / (R * th * np.exp(N * N * z / g))


def states(sem, m, eqset):
    xyz = sem.sem_mesh_coords_host(m).T
    base = random_state(xyz, LZ, 5, "C" if eqset == 0 else "NC")
    rng = np.random.default_rng(1)
    yield "random", base
    yield "rest", np.zeros_like(base)
    q = np.zeros_like(base)
    q[1] = 7.5
    yield "uniform", q   # every node of an element is a candidate
    q = base.copy()
    q[1:4] *= 1e-30
    q[1:4, ::3] = 0.0
    yield "tiny", q
    q = base * 10.0 ** rng.uniform(-25, 5, size=base.shape[1])[None]
    yield "scales", q
    q = base.copy()
    q[2, rng.integers(0, m.NG, 20)] = np.nan
    q[3, rng.integers(0, m.NG, 20)] = np.inf
    q[1, rng.integers(0, m.NG, 20)] = -1e30
    q[0, rng.integers(0, m.NG, 20)] = -2.0   # a density below zero
    yield "special", q


@pytest.mark.parametrize("eqset", [0, 1])
@pytest.mark.parametrize("N,nz", [(2, 3), (3, 1), (3, 90), (4, 16), (4, 63), (4, 64), (5, 7), (6, 43)])
def test_speed_criterion_bits(sem, N, nz, eqset):
    m = make(sem, N, nz)
    thr = [5.0, 10.0, 15.0]
    p = sem.sem_params_default(thresholds=thr, lvl_max=3, eqset=eqset)
    lev = np.repeat(sem.sem_mesh_leaves_host(m)[:, 0], nz)
    z = sem.sem_mesh_coords_host(m)[2].reshape(m.NH, m.NZ)[0]
    for name, q in states(sem, m, eqset):
        L = local_lines(sem, m, q)
        with np.errstate(all="ignore"):
            s = np.sqrt(L[1] * L[1] + L[2] * L[2] + L[3] * L[3])
            if eqset == 0:
                s = s / (background_rho(z) + L[0])
        el = np.stack([s[:, :, k * N:k * N + N + 1] for k in range(nz)], axis=1).reshape(m.Ne, -1)
        want = np.fmax.reduce(el, axis=1)
        if (N + 1) ** 3 % 32:
            want = np.fmax(want, 0.0)
        flags = torch.empty(m.Ne, dtype=torch.int8, device="cuda")
        cmax = torch.empty(m.Ne, dtype=torch.float64, device="cuda")
        sem.sem_adapt_flags(m, p, torch.from_numpy(q).cuda(), flags, cmax)
        got = cmax.cpu().numpy()
        # the reference density differs from the library's table by rounding
        if eqset == 1:
            np.testing.assert_array_equal(got, want, err_msg=name)
        else:
            fin = np.isfinite(want)
            np.testing.assert_array_equal(np.isfinite(got), fin, err_msg=name)
            ok = fin if name != "special" else fin & (np.nanmin(np.abs(background_rho(z)[None, None] + L[0])) > 0)
            np.testing.assert_allclose(got[ok], want[ok], rtol=1e-12 if name != "special" else 1e-9, err_msg=name)
        with np.errstate(invalid="ignore"):
            up = (lev < 3) & (got > np.array(thr)[np.minimum(lev, 2)])
            down = (lev > 0) & (got <= np.array(thr)[np.maximum(lev - 1, 0)])
        np.testing.assert_array_equal(flags.cpu().numpy(), np.where(up, 1, np.where(down, -1, 0)), err_msg=name)


@pytest.mark.parametrize("N,nz,n,half", [(4, 3, 4, 40e3), (4, 100, 3, 150e3), (3, 5, 9, 75e3), (6, 1, 4, 10e3), (2, 3, 40, 60e3),
                                         (4, 100, 18, 20e3), (3, 11, 24, 150e3)])
def test_diag_levels(sem, N, nz, n, half):
    """Levels within, across and beyond one block of threads; the node list
    across several blocks."""
    m = make(sem, N, nz, n)
    xyz = sem.sem_mesh_coords_host(m)
    q = random_state(xyz.T, LZ, 8)
    d = sem.sem_diag(m, sem.sem_params_default(), torch.from_numpy(q).cuda(), half)
    near = (np.abs(xyz[0]) <= half + 1e-6) & (np.abs(xyz[1]) <= half + 1e-6)
    s = np.sqrt(q[1] ** 2 + q[2] ** 2) / (background_rho(xyz[2]) + q[0])
    w = sem.sem_mesh_mass_host(m) * near
    num, den = (w * s).reshape(-1, m.NZ).sum(0), w.reshape(-1, m.NZ).sum(0)
    assert abs(d["max_wind"] / s[near].max() - 1) < 1e-12
    assert abs(d["max_mean_wind"] / (num / den).max() - 1) < 1e-12


@pytest.mark.parametrize("N,nz", [(2, 17), (3, 5), (4, 16), (4, 17), (5, 33), (6, 2)])
def test_features_orders(sem, N, nz):
    """Every order, layer counts around the chunk, hanging lines; values from
    zeros and float32's denormals to its largest, and odd scales.  The quotient
    is rounded to float32 to within one unit in the last place."""
    m = make(sem, N, nz)
    o = om.OracleMesh(300e3, 300e3, LZ, 4, 4, nz, N, leaves=two_level(4))
    perm = node_perm(sem.sem_mesh_coords_host(m), o.XG)
    q = random_state(o.XG, LZ, 4)
    rng = np.random.default_rng(2)
    spread = q * 10.0 ** rng.uniform(-60, 25, size=q.shape)
    spread[:, ::5] = 0.0
    for data, scales in ((q, (1e-3, 10.0, 7.0, 1.0, -3.0)), (spread, (1e-3, 3e7, 1e-9, 1.0, 1.7))):
        want = omlp.features(o, data, np.asarray(scales, np.float32).astype(np.float64))
        F = torch.empty((m.Ne, 136), dtype=torch.float32, device="cuda")
        sem.sem_mlp_features(m, torch.from_numpy(np.ascontiguousarray(data[:, perm])).cuda(), scales, F)
        oleaf = {tuple(l): c for c, l in enumerate(o.leaves)}
        emap = np.array([oleaf[tuple(l)] * nz + k for l in sem.sem_mesh_leaves_host(m) for k in range(nz)])
        got, want = F.cpu().numpy().astype(np.float64), want[emap]
        # interpolated values carry the cancellation of their terms
        lvl = 0.0 if N % 2 == 0 and data is q else 1e-13 * np.abs(want).max()
        assert np.all(np.abs(got - want) <= 1.2e-7 * np.abs(want) + 1.5e-45 + lvl)


@pytest.mark.parametrize("N,nz", [(2, 3), (3, 13), (4, 1), (4, 12), (5, 4), (6, 2)])
def test_transfer_orders(sem, N, nz):
    """Refined, coarsened and unchanged columns together, from a 2:1 mesh,
    against the oracle: one and several passes over a column's levels."""
    m = make(sem, N, nz)
    o = om.OracleMesh(300e3, 300e3, LZ, 4, 4, nz, N, leaves=two_level(4))
    perm = node_perm(sem.sem_mesh_coords_host(m), o.XG)
    q_o = random_state(o.XG, LZ, 9)
    q = torch.from_numpy(np.ascontiguousarray(q_o[:, perm])).cuda()
    for change in ({(0, 3, 3): 1, (0, 0, 2): 1}, {(1, 2 + a, 2 + b): -1 for a in (0, 1) for b in (0, 1)},
                   {(1, 2, 2): 1}):
        lv = [tuple(l) for l in sem.sem_mesh_leaves_host(m).tolist()]
        fl = np.repeat(np.array([change.get(l, 0) for l in lv], dtype=np.int8), nz)
        fl_o = np.zeros(o.Ne, dtype=np.int8)
        for c, l in enumerate(o.leaves):
            fl_o[c * nz:(c + 1) * nz] = change.get(tuple(l), 0)
        new = sem.sem_transfer_plan(m, fl)
        new_o, org = adapt.update_leaves(o.leaves, fl_o, nz, 4, 4, 3)
        o2, want = otr.transfer(o, new_o, org, q_o)
        perm2 = node_perm(sem.sem_mesh_coords_host(new), o2.XG)
        got = torch.empty(5, new.NG, dtype=torch.float64, device="cuda")
        sem.sem_transfer(m, new, q, got)
        err = np.linalg.norm(got.cpu().numpy() - want[:, perm2], axis=1) / np.linalg.norm(want, axis=1)
        assert np.all(err <= 1e-12), (change, err)
        assert sem.sem_status(new) == 0
