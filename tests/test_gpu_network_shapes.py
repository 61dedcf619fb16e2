"""The closure network's kernels (four threads per sample) at the edges of their
shapes."""
import numpy as np
import pytest

from oracle import closure as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_01287_gb300 import build, load
    build.build()
    load()


def _as_used(theta, D, H, O):
    """BF16 weights, FP32 biases, FP64."""
    out, o = [], 0
    for k, n in enumerate(C.param_sizes(D, H, O)):
        part = theta[o:o + n]
        out.append(C.bf16_round(part) if k % 2 == 0 else part.astype(np.float64))
        o += n
    return np.concatenate(out)


@pytest.mark.parametrize("D,H,O", [(128, 64, 32), (7, 16, 1), (97, 32, 9), (73, 64, 24)])
@pytest.mark.parametrize("n", [1, 63, 129, 1000])
def test_forward_and_gradient(D, H, O, n):
    """FP32 sums of at most 128 terms (samples are summed over CTAs too): 1e-5 of the
    largest value."""
    import torch
    from paper_1612_01287_gb300 import MLP
    rng = np.random.default_rng(D + n)
    X = rng.normal(size=(n, D)).astype(np.float32)
    T = rng.normal(size=(n, O)).astype(np.float32)
    theta = rng.normal(0, 0.3 / np.sqrt(H), size=sum(C.param_sizes(D, H, O))).astype(np.float32)
    Xd, Td = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
    Y = torch.empty((n, O), device="cuda")
    with MLP(D, H, O) as m:
        m.set_params(theta)
        m.forward(Xd.data_ptr(), n, Y.data_ptr())
        torch.cuda.synchronize()
        loss, g = m.loss_grad(Xd.data_ptr(), Td.data_ptr(), n)
    th = _as_used(theta, D, H, O)
    y, _ = C.forward(th, X.astype(np.float64), D, H, O)
    L, gr = C.loss_grad(th, X.astype(np.float64), T.astype(np.float64), D, H, O)
    assert np.abs(Y.cpu().numpy() - y).max() <= 1e-5 * np.abs(y).max()
    assert abs(loss - L) <= 1e-5 * L
    assert np.abs(g - gr).max() <= 1e-5 * np.abs(gr).max()


@pytest.mark.parametrize("Z,Q_xi,Q_L,hidden", [(65, 4, 2, 16), (200, 8, 3, 64), (130, 16, 2, 32)])
def test_closure_steps_of_any_count_agree(Z, Q_xi, Q_L, hidden):
    """The state changes buffers every step: three steps at once, two and one, and
    three single calls leave bitwise the same state, which rslb_step continues."""
    from paper_1612_01287_gb300 import MLP, Sod, closure_step
    V = Q_xi * Q_L
    out = []
    for parts in ([3], [2, 1], [1, 1, 1]):
        with Sod(Z=Z, Q_xi=Q_xi, Q_L=Q_L, precision="f32", bc="outflow", tau=0.05, dt=1e-3) as s, \
                MLP(3 * V + 1, hidden, V, seed=5) as m:
            m.set_normalization(np.zeros(3 * V + 1), np.ones(3 * V + 1), np.full(V, 1e-3))
            for n in parts:
                closure_step(s, m, 0.05, n)
            s.step(2)
            out.append(s.get_state())
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])
