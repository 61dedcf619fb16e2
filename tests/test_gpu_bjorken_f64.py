"""The FP64 Bjorken kernel (even/odd half-size matrices) at the edges of its
blocking: the smallest Q_xi, odd and even ones, one and eight radial nodes, and
more runs of one Q_xi than one per block."""
import math

import numpy as np
import pytest

from tests.test_gpu_bjorken import oracle_batch, errors, run_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1612_01287_gb300 import build, load
    build.build()
    load()


@pytest.mark.parametrize("Q_L", [1, 2, 8])
@pytest.mark.parametrize("Qs", [[2], [3], [31, 32, 33, 2, 33], [200, 201]])
def test_small_odd_and_even_orders(Qs, Q_L):
    """FP64 parity (1e-12, the suite's bound) with the oracle."""
    gases = ["parton" if i % 2 else "ideal" for i in range(len(Qs))]
    taus = [0.2 if i % 3 else math.inf for i in range(len(Qs))]
    got, state = run_batch(Qs, gases, taus, "f64", 10, Q_L=Q_L)
    ref, rstates = oracle_batch(Qs, gases, taus, 10, Q_L=Q_L)
    for k, v in errors(got, ref).items():
        assert v <= 1e-12, (k, v)
    flat = np.concatenate(rstates)
    assert np.abs(state - flat).max() <= 1e-12 * np.abs(flat).max()


def test_blocks_of_several_runs():
    """Enough equal runs that a block holds several: each is bitwise the run alone."""
    from paper_1612_01287_gb300 import Bjorken
    taus = np.linspace(0.05, 2.0, 4000)
    with Bjorken([12] * len(taus), "parton", taus, Q_L=2, precision="f64", dtau=1e-2) as b:
        b.step(5)
        many = b.get_state().reshape(len(taus), -1)
    for r in (0, 1, 1777, 3999):
        with Bjorken([12], "parton", [taus[r]], Q_L=2, precision="f64", dtau=1e-2) as b:
            b.step(5)
            np.testing.assert_array_equal(b.get_state(), many[r])
