"""The network's features value by value.

A feature that is a node's value (even orders, nodes of the mesh) is
(float)(v / s) of the float64 quotient, bit for bit: quotients next to the
midpoint between two float32 numbers, from below float32's smallest value to
beyond its largest, zeros of both signs, infinities and NaN.  Interpolated ones
carry the rounding of their terms."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import basis  # noqa: E402
from synth.vortex import random_state  # noqa: E402
from tests.test_gpu_remesh import LZ, local_lines, make  # noqa: E402

SCALES = (1e-3, 10.0, 7.0, 1e-9, -3.0)


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


def features(sem, m, q, scales):
    F = torch.full((m.Ne, 136), float("nan"), dtype=torch.float32, device="cuda")
    sem.sem_mlp_features(m, torch.from_numpy(np.ascontiguousarray(q)).cuda(), scales, F)
    return F.cpu().numpy()[:, :135].reshape(m.Ncol, m.nz, 5, 3, 3, 3)   # [.., field, c, b, a]


def node_values(kind, shape, s, rng):
    """Values v [5, n] per scale: midpoints of neighbouring float32 quotients
    moved by up to two units of v, or a wide range of magnitudes."""
    out = np.empty(shape)
    for f in range(5):
        if kind == "midpoints":
            a = (rng.integers(0x3F000000, 0x43000000, shape[1]).astype(np.uint32)).view(np.float32)
            mid = 0.5 * (a.astype(np.float64) + np.nextafter(a, np.float32(np.inf)).astype(np.float64))
            v = mid * s[f] * rng.choice([-1.0, 1.0], shape[1])
            out[f] = (v.view(np.int64) + rng.integers(-2, 3, shape[1])).view(np.float64)
        else:
            out[f] = rng.uniform(-2, 2, shape[1]) * 10.0 ** rng.uniform(-60, 45, shape[1])
            out[f, ::7] = 0.0
            out[f, 1::7] *= 0.0   # zeros of either sign
    return out


@pytest.mark.parametrize("N,nz", [(2, 3), (4, 17)])
@pytest.mark.parametrize("kind", ["midpoints", "wide"])
def test_node_values_are_the_rounded_quotient(sem, N, nz, kind):
    m = make(sem, N, nz, 12, leaves=[(0, i, j) for i in range(12) for j in range(12)])
    s = np.asarray(SCALES, np.float32).astype(np.float64)
    q = node_values(kind, (5, m.NG), s, np.random.default_rng(3))
    if kind == "wide":
        q[:, 5::1001], q[:, 6::1001], q[:, 8::1001] = np.nan, np.inf, -np.inf
    got = features(sem, m, q, SCALES)
    with np.errstate(all="ignore"):
        want = (local_lines(sem, m, q) / s[:, None, None, None]).astype(np.float32)
    n1, h = N + 1, N // 2
    for k in range(nz):
        for c in range(3):
            for b in range(3):
                for a in range(3):
                    w = want[:, :, a * h + n1 * b * h, k * N + c * h].T
                    g = got[:, k, :, c, b, a]
                    nan = np.isnan(w)
                    np.testing.assert_array_equal(np.isnan(g), nan)
                    np.testing.assert_array_equal(g.view(np.int32)[~nan], w.view(np.int32)[~nan])


@pytest.mark.parametrize("N,nz", [(2, 17), (3, 5), (4, 16), (5, 33), (6, 2)])
def test_interpolated_values_within_their_terms(sem, N, nz):
    """Every order and hanging lines, values over 85 decades: half a unit of
    float32, and for each side's float64 sums one rounding of the sum of the
    absolute terms per link of the longest chain: N + 1 terms of a hanging line,
    (N + 1)^2 in the plane, N + 1 along z, and the weights' own (8)."""
    m = make(sem, N, nz)
    X = sem.sem_mesh_coords_host(m).T
    rng = np.random.default_rng(2)
    q = random_state(X, LZ, 4) * 10.0 ** rng.uniform(-60, 25, size=(5, m.NG))
    q[:, ::5] = 0.0
    s = np.asarray(SCALES, np.float32).astype(np.float64)
    got = features(sem, m, q, SCALES).astype(np.float64)
    n1 = N + 1
    H = basis.lagrange_eval(basis.lgl_nodes_weights(N)[0], np.array([-1.0, 0.0, 1.0]))
    H[0], H[2] = np.eye(n1)[0], np.eye(n1)[N]
    if N % 2 == 0:
        H[1] = np.eye(n1)[N // 2]
    hmap, hh, hw = sem.sem_mesh_hmap_host(m)
    for H_, vals in ((H, q), (np.abs(H), np.abs(q))):
        w = hw if H_ is H else np.abs(hw)
        v = vals.reshape(5, m.NH, m.NZ)
        hang = np.einsum("hm,fhmz->fhz", w, v[:, hh])
        L = np.where(hmap[None, :, :, None] >= 0, v[:, np.maximum(hmap, 0)], hang[:, np.maximum(-1 - hmap, 0)])
        L = L.reshape(5, m.Ncol, n1, n1, m.NZ)
        L = np.stack([L[..., k * N:k * N + n1] for k in range(nz)], axis=4)   # [f, col, b, a, k, c]
        T = np.einsum("Aa,Bb,Cc,fobakc->okfCBA", H_, H_, H_, L)
        if H_ is H:
            want = T / s[None, None, :, None, None, None]
        else:
            terms = T / np.abs(s)[None, None, :, None, None, None]
    big = np.abs(want) > 3.4e38
    assert np.all(np.abs(got[big]) >= 3.4e38)
    err = np.abs(got - want)[~big]
    chain = 2 * (n1 * n1 + 2 * n1 + 8) * 2.0 ** -53
    assert np.all(err <= 2.0 ** -24 * np.abs(want[~big]) + 1.001 * chain * terms[~big] + 2.0 ** -150)
