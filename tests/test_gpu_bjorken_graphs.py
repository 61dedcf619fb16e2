"""Tensor-core Bjorken steps in graphs of eight and of two and as plain launches."""
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


@pytest.mark.parametrize("parts", [(8, 8, 9), (1, 8, 16), (19, 3, 2, 1), (2, 23), (7, 17, 1),
                                   (1, 2, 3, 4, 5, 6, 4)])
def test_step_counts(parts):
    """25 steps in any parts, from either parity of the moment buffers, give bitwise the
    states of plain launches (the default stream)."""
    import torch
    from paper_1612_01287_gb300 import Bjorken
    assert sum(parts) == 25
    Qs, gases, taus = [64, 8, 200, 64], ["parton", "ideal", "parton", "ideal"], [0.1, 0.5, 2.0, np.inf]
    kw = dict(Q_L=2, precision="f32", kp_mode="tf32x3", dtau=1e-2)
    with Bjorken(Qs, gases, taus, **kw) as a, \
            Bjorken(Qs, gases, taus, stream=torch.cuda.Stream(), **kw) as b:
        a.step(25)
        for n in parts:
            b.step(n)
        fa, fb, ra, rb = a.get_state(), b.get_state(), a.read(), b.read()
    np.testing.assert_array_equal(fa, fb)
    for k in ra:
        np.testing.assert_array_equal(ra[k], rb[k])
