"""Output moments at radial sets and cell counts that leave ragged blocks and
chunks."""
import numpy as np
import pytest

import oracle
from tests import sodcase

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_01287_gb300 import build, load
    build.build()
    load()


@pytest.mark.parametrize("precision,tol", [("f64", 1e-13), ("f32", 1e-12)])
@pytest.mark.parametrize("Z,Q_xi,Q_L", [(1, 3, 1), (63, 4, 8), (65, 33, 2), (130, 200, 3)])
def test_output_moments_shapes(precision, tol, Z, Q_xi, Q_L):
    """Into device memory (written by the kernel) and into host memory, against the
    oracle on the stored populations (the suite's bounds)."""
    import torch
    from paper_1612_01287_gb300 import Sod
    z = (np.arange(Z) + 0.5) / Z
    fields = (1 + 0.3 * np.sin(5 * z), 1 + 0.2 * np.cos(4 * z), 0.5 * np.sin(3 * z))
    case = dict(Z=Z, Q_xi=Q_xi, Q_L=Q_L, bc="outflow", tau=1e-2, dt=1e-4)
    with Sod(precision=precision, fields=fields, **case) as s:
        host = s.moments()
        dev = torch.zeros((14, Z), dtype=torch.float64, device="cuda")
        s.moments(out=dev)
        off = torch.zeros(14 * Z * 8 + 4, dtype=torch.uint8, device="cuda")[4:]  # not 8-byte aligned
        s.moments(out=off)
        f = s.get_state().astype(np.float64)
    a = np.stack(list(host.values()))
    np.testing.assert_array_equal(a, dev.cpu().numpy())
    np.testing.assert_array_equal(a.tobytes(), off.cpu().numpy()[:14 * Z * 8].tobytes())
    mo = oracle.sod_moments(sodcase.oracle_params(case), np.ascontiguousarray(f.T))
    for k in ("n", "E", "beta", "Pi", "Nt", "Nz", "Ttt", "Ttz", "Tzz"):
        assert np.abs(host[k] - mo[k]).max() <= tol * max(1.0, np.abs(mo["E"]).max()), k
