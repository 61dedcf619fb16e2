"""The populations of a tensor-core Bjorken batch come back in the callers' order:
runs out of order, populations per run below, at and above the copying block
(256 threads) and the smallest and largest Q_xi of the workload."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_01287_gb300 import build, load
    build.build()
    load()


@pytest.mark.parametrize("Q_L", [1, 2, 3])
@pytest.mark.parametrize("Qs", [[8], [85, 512, 9, 86, 8, 86], [128, 256, 129, 255, 257, 127]])
def test_state_returns_in_the_callers_order(Qs, Q_L):
    """set_state then get_state is bitwise the same, and stays so after K^P f, which
    is read through the same scratch buffer."""
    from paper_1612_01287_gb300 import Bjorken
    f = np.random.default_rng(sum(Qs) + Q_L).uniform(0.1, 1.0, Q_L * sum(Qs)).astype(np.float32)
    with Bjorken(Qs, "parton", 0.2, Q_L=Q_L, precision="f32", kp_mode="tf32x3", dtau=1e-3) as b:
        b.set_state(f)
        np.testing.assert_array_equal(b.get_state(), f)
        b.kp_apply()
        np.testing.assert_array_equal(b.get_state(), f)
