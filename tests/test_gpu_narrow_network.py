"""Networks of 16 or 32 hidden units and few inputs: one thread per sample from many
samples on, four below; gradients over more partials than one round of the sum."""
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


@pytest.mark.parametrize("D,H,O,n", [
    (1, 16, 1, 49151), (1, 16, 1, 49152), (32, 16, 32, 49185), (31, 16, 10, 90001),
    (33, 16, 32, 49185), (2, 32, 1, 327679), (2, 32, 1, 327711), (32, 32, 32, 327681)])
def test_forward(D, H, O, n):
    """FP32 sums of at most 33 terms: 1e-5 of the largest value."""
    import torch
    from paper_1612_01287_gb300 import MLP
    rng = np.random.default_rng(D + n)
    X = rng.normal(size=(n, D)).astype(np.float32)
    theta = rng.normal(0, 0.4, size=sum(C.param_sizes(D, H, O))).astype(np.float32)
    Xd = torch.tensor(X, device="cuda")
    Y = torch.full((n + 1, O), np.nan, device="cuda")
    with MLP(D, H, O) as m:
        m.set_params(theta)
        m.forward(Xd.data_ptr(), n, Y.data_ptr())
        torch.cuda.synchronize()
    y, _ = C.forward(_as_used(theta, D, H, O), X.astype(np.float64), D, H, O)
    got = Y.cpu().numpy()
    assert np.abs(got[:n] - y).max() <= 1e-5 * np.abs(y).max()
    assert np.isnan(got[n]).all()


@pytest.mark.parametrize("H", [16, 32])
@pytest.mark.parametrize("Q_xi,Q_L,Z", [(2, 2, 49151), (2, 2, 49152), (5, 2, 49185)])
def test_closure_step(Q_xi, Q_L, Z, H):
    """One step against the FP64 correction of the stepped state: 1e-5 of its maximum."""
    from paper_1612_01287_gb300 import MLP, Sod, closure_step
    V, tau = Q_xi * Q_L, 0.05
    z = (np.arange(Z) + 0.5) / Z
    fields = (1.0 + 0.3 * np.sin(700 * z) + (z > 0.4), 1.0 + 0.2 * np.cos(500 * z),
              0.4 * np.sin(900 * z + 1))
    kw = dict(Z=Z, Q_xi=Q_xi, Q_L=Q_L, precision="f32", bc="outflow", tau=tau, dt=0.5 / Z,
              fields=fields)
    D = 3 * V + 1
    rng = np.random.default_rng(V + H)
    norm = (rng.normal(0, 0.1, D).astype(np.float32), rng.uniform(0.5, 2, D).astype(np.float32),
            rng.uniform(0.5e-2, 2e-2, V).astype(np.float32))
    with MLP(D, H, V, seed=5) as m, Sod(**kw) as a, Sod(**kw) as c:
        th = m.get_params()
        th[D * H + H + H * H + H:] *= 10.0  # a visible correction
        m.set_params(th)
        m.set_normalization(*norm)
        a.step(1)
        closure_step(c, m, tau, 1)
        fa, fc = (x.get_state().astype(np.float64).T for x in (a, c))
        thr = _as_used(m.get_params(), D, H, V)
    ref = C.correction(thr, fa, tau, Q_xi, Q_L, H, tuple(x.astype(np.float64) for x in norm))
    assert np.abs(ref).max() > 1e-4 * np.abs(fa).max()
    assert np.abs((fc - fa) - ref).max() <= 1e-5 * np.abs(fa).max()


@pytest.mark.parametrize("n", [128 * 127 + 1, 128 * 128 + 1, 128 * 257])
@pytest.mark.parametrize("D,H,O", [(1, 16, 1), (20, 32, 5)])
def test_gradient_over_many_partials(D, H, O, n):
    """FP32 sums of the samples in blocks of 128, then of the blocks: 1e-5 of the
    largest entry; twice the same bits."""
    import torch
    from paper_1612_01287_gb300 import MLP
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, D)).astype(np.float32)
    T = (X[:, :1] + rng.normal(size=(n, O))).astype(np.float32)
    theta = rng.normal(0, 0.4, size=sum(C.param_sizes(D, H, O))).astype(np.float32)
    Xd, Td = torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda")
    with MLP(D, H, O) as m:
        m.set_params(theta)
        loss, g = m.loss_grad(Xd.data_ptr(), Td.data_ptr(), n)
        loss2, g2 = m.loss_grad(Xd.data_ptr(), Td.data_ptr(), n)
    L, gr = C.loss_grad(_as_used(theta, D, H, O), X.astype(np.float64), T.astype(np.float64), D, H, O)
    assert abs(loss - L) <= 1e-6 * L
    assert np.abs(g - gr).max() <= 1e-5 * np.abs(gr).max()
    assert loss == loss2 and np.array_equal(g, g2)
