"""The network's passes at the edges of their tiles of rows, of the splits of the
gradient sums and of the persistent blocks, for both forwards: gradients against
float64 on inputs whose hidden activations are exact in bfloat16 or rounded from
exact sums, so that no rounding of an activation can fall differently."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CW = (0.6, 0.5, 4.0)


@pytest.fixture(scope="module")
def sem():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_21607_gb300 import build
    build.build()
    from paper_2410_21607_gb300 import sem as s
    return s


def bf16(x):
    return x.float().bfloat16().double()


def case(sem, n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randint(-2, 3, (n, 136), generator=g, device="cuda").float()
    net = sem.sem_mlp_create(seed, n)
    p = (np.round(sem.sem_mlp_get_params(net) * 64) / 64).astype(np.float32)
    sem.sem_mlp_set_params(net, p)
    y = torch.randint(0, 3, (n,), generator=g, device="cuda").to(torch.int8)
    P, at, W = torch.from_numpy(p).cuda().double(), 0, []
    for a, b in ((136, 128), (128, 128), (128, 3)):
        W += [P[at:at + a * b].reshape(a, b), P[at + a * b:at + a * b + b]]
        at += a * b + b
    Xd = X.double()
    H1 = bf16(torch.relu(Xd @ W[0] + W[1]))
    H2 = bf16(torch.relu(H1 @ W[2] + W[3]))
    prob = torch.softmax(H2 @ W[4] + W[5], 1)
    w = torch.tensor(CW, device="cuda").double()[y.long()]
    d3 = (w / w.sum())[:, None] * (prob - torch.nn.functional.one_hot(y.long(), 3))
    d2 = (d3 @ W[4].T) * (H2 > 0)
    d1 = (d2 @ W[2].T) * (H1 > 0)
    grads = [Xd.T @ d1, d1.sum(0), H1.T @ d2, d2.sum(0), H2.T @ d3, d3.sum(0)]
    loss = float((w * -torch.log(prob[torch.arange(n), y.long()])).sum() / w.sum())
    return X, y, net, prob, grads, loss


@pytest.mark.parametrize("tc", [1, 0])
@pytest.mark.parametrize("n", [1, 7, 127, 128, 129, 1023, 1025, 152 * 128 + 1, 40000])
def test_gradients_at_tile_edges(sem, n, tc):
    """Every parameter block within 8 units of float32 rounding of its norm (the
    probabilities carry exp's and the quotient's error, a gradient's terms
    partly cancel); the same bits on every call."""
    X, y, net, prob, want, loss = case(sem, n, n % 1000)
    sem.sem_mlp_select_forward(net, tc)
    got_loss = sem.sem_mlp_backward(net, X, y, CW)
    got = torch.from_numpy(sem.sem_mlp_get_grads(net)).cuda().double()
    at = 0
    for g in want:
        e = (got[at:at + g.numel()] - g.reshape(-1)).norm() / max(float(g.norm()), 1e-30)
        scale = float(want[-1].abs().sum()) if g.numel() == 3 else 0.0   # sums to zero over the classes
        assert float(e) <= 8 * 2.0 ** -23 or (g.numel() == 3 and scale < 1e-3), (n, at, float(e))
        at += g.numel()
    assert abs(got_loss / loss - 1) < 1e-6
    # the same bits again, and without the loss
    sem.sem_mlp_backward(net, X, y, CW, want_loss=False)
    np.testing.assert_array_equal(sem.sem_mlp_get_grads(net), got.cpu().numpy().astype(np.float32))
    p = torch.empty((n, 3), device="cuda")
    sem.sem_mlp_forward(net, X, p)
    assert float((p.double() - prob).abs().max()) < 1e-6
    assert sem.sem_mlp_status(net) == 0


def test_backward_of_a_row_at_any_address(sem):
    """The mma.sync forward takes inputs at any 4-byte address; so does the
    backward pass behind it."""
    X, y, net, prob, want, _ = case(sem, 200, 5)
    sem.sem_mlp_select_forward(net, 0)
    sem.sem_mlp_backward(net, X, y, CW)
    a = sem.sem_mlp_get_grads(net)
    shifted = torch.empty(X.numel() + 1, device="cuda")[1:].view(X.shape)
    shifted.copy_(X)
    assert shifted.data_ptr() % 16 == 4
    sem.sem_mlp_backward(net, shifted, y, CW)
    np.testing.assert_array_equal(sem.sem_mlp_get_grads(net), a)
