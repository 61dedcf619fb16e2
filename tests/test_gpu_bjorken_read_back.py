"""Populations of Bjorken batches in the callers' order by each of the three ways: as they
lie, reordered on the host, gathered on the device (tensor-core batches from 128 KB on)."""
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


RISING = [8, 9, 100, 511, 512]
# 32768 FP32 values are the 128 KB
CASES = [[64], [512, 100, 100, 8], RISING, RISING * 9, sorted(RISING * 12, reverse=True),
         [300] * 36 + [122], [122] + [300] * 36, [300] * 36 + [123], [123] + [300] * 36]


@pytest.mark.parametrize("kp_mode,precision", [("tf32x3", "f32"), ("simt", "f32"), ("simt", "f64")])
@pytest.mark.parametrize("Qs", CASES, ids=lambda q: "%d-%d" % (len(q), sum(q)))
def test_state_comes_back(Qs, kp_mode, precision):
    """set_state then get_state gives the same bits, on the default stream and on another,
    and after K^P f has gone through the same buffers; K^P f of a run does not depend on
    the way it came."""
    import torch
    from paper_1612_01287_gb300 import Bjorken
    dtype = np.float32 if precision == "f32" else np.float64
    f = np.random.default_rng(sum(Qs)).uniform(0.1, 1.0, 3 * sum(Qs)).astype(dtype)
    kw = dict(Q_L=3, precision=precision, kp_mode=kp_mode, dtau=1e-3)
    for stream in (None, torch.cuda.Stream()):
        with Bjorken(Qs, "parton", 0.2, stream=stream, **kw) as b:
            b.set_state(f)
            np.testing.assert_array_equal(b.get_state(), f)
            if kp_mode == "simt":
                continue
            y = b.kp_apply()
            np.testing.assert_array_equal(b.get_state(), f)
        with Bjorken(Qs[:1], "parton", 0.2, stream=stream, **kw) as b:
            b.set_state(f[:3 * Qs[0]])
            alone = b.kp_apply()
        scale = np.abs(alone).max()
        assert np.abs(y[:3 * Qs[0]] - alone).max() <= 1e-5 * scale
