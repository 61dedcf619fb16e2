"""f^eq of fast flows in the stage kernels.  A uniform beam f = w_j w_k e^{a (xi_j - 1)}
(f > 0, so its moments resolve the flow in FP32 too, which those of a truncated
equilibrium at |beta| near 1 do not) relaxes for one step; the flux vanishes, so
what is left is the relaxation towards f^eq at the beam's (n, T, beta).  Faster
beams are non-physical after one stage, because the truncated f^eq is negative
against the flow; the coefficients beyond are compared on the CPU."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_01287_gb300 import build, load
    build.build()
    load()


@pytest.mark.parametrize("precision,Q_xi,Q_L,N_Omega,tile", [
    ("f32", 200, 3, 5, 28), ("f32", 200, 3, 7, 28), ("f32", 200, 3, 5, 32),
    ("f32", 200, 3, 12, 0), ("f32", 100, 1, 3, 64), ("f64", 200, 3, 5, 0),
    ("f64", 200, 3, 12, 8), ("f64", 200, 1, 12, 16)])
@pytest.mark.parametrize("a,beta,x", [(2, 0.44, 1e-2), (8, 0.83, 1e-2), (20, 0.93, 1e-2),
                                      (40, 0.965, 1e-3)])
@pytest.mark.parametrize("sign", [1, -1])
def test_beam_relaxes_to_its_equilibrium(precision, Q_xi, Q_L, N_Omega, tile, a, beta, x, sign):
    """Roundings of the moments (products, blocks, weights: <= 8 eps of a positive
    sum) pass into gamma and f^eq with factors of order one, and the coefficients
    add <= 20 eps (64 in the 32-node rule): 100 eps of the populations and of
    their change."""
    from paper_1612_01287_gb300 import Sod
    Z, tau = 40, 2e-2
    dt = x * tau
    xi, w, xk, wk = oracle.gauss_legendre(Q_xi) + oracle.gauss_laguerre2(Q_L)
    f = (wk[:, None] * w[None, :] * np.exp(a * (sign * xi - 1.0))[None, :]).ravel()
    dtype = np.float32 if precision == "f32" else np.float64
    f = np.repeat(f.astype(dtype)[:, None], Z, axis=1)
    lan = oracle.landau(oracle.moments(Q_xi, Q_L, f[:, 0].astype(np.float64)))
    assert abs(lan["beta"] - sign * beta) < 0.005
    p = oracle.sod_params(Z, Q_xi, Q_L, N_Omega, bc="outflow", tau=tau, dt=dt)
    ref = oracle.sod_steps(p, f.T.astype(np.float64), 1).T
    with Sod(Z=Z, Q_xi=Q_xi, Q_L=Q_L, N_Omega=N_Omega, precision=precision, bc="outflow",
             tau=tau, dt=dt, tile_cells=tile) as s:
        s.set_state(f)
        s.step(1)
        got = s.get_state()
    change = np.abs(ref - f).max()
    assert change > 0.1 * x * np.abs(f).max()
    eps = float(np.finfo(dtype).eps)
    assert np.abs(got - ref).max() <= 100 * eps * (np.abs(f).max() + change)
