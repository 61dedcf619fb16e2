"""Batches of one velocity class take every place the SMs have for their kernel, and
give bitwise what they give beside other classes."""
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


def _runs(Q_xi, n, Z):
    return [dict(Z=Z + 17 * i, Q_xi=Q_xi, tau=0.05, dt=0.2 / Z, t_end=1.6 / Z) for i in range(n)]


def _fields(runs, precision, n):
    from paper_1612_01287_gb300 import SodBatch
    with SodBatch(runs, Q_L=3, precision=precision, autotune=False) as b:
        b.step(8)
        return b.tuning(), [np.stack(list(b.moments(r).values())) for r in range(n)]


@pytest.mark.parametrize("precision,Q_xi,tile,places", [
    ("f32", 50, 28, 3), ("f32", 100, 28, 3), ("f32", 200, 28, 2), ("f32", 8, 128, 2),
    ("f64", 20, 16, 2)])
@pytest.mark.parametrize("n,Z", [(1, 40), (16, 1000)])
def test_one_class(precision, Q_xi, tile, places, n, Z):
    """Fewer tiles than places, and more."""
    runs = _runs(Q_xi, n, Z)
    tuning, alone = _fields(runs, precision, n)
    assert tuning == [(3 * Q_xi, tile, places)]
    _, beside = _fields(runs + _runs(6, 2, 300), precision, n)
    for a, b in zip(alone, beside):
        np.testing.assert_array_equal(a, b)
