"""Batches with more velocity classes than concurrent chains."""
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


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("classes", [15, 16, 17, 37])
def test_more_classes_than_chains(precision, classes):
    """Plain launches and graph replays give bitwise the fields of every class as a
    batch of its own."""
    import torch
    from paper_1612_01287_gb300 import SodBatch
    runs = [dict(Z=60 + 11 * q, Q_xi=3 + q, tau=0.05, dt=1e-4 * (1 + q % 3), t_end=2e-3)
            for q in range(classes)]
    kw = dict(Q_L=2, precision=precision, autotune=False, stream=torch.cuda.Stream())
    with SodBatch(runs, **kw) as b:
        for n in (3, 16, 2):
            b.step(n)
        got = [np.stack(list(b.moments(r).values())) for r in range(classes)]
    for run, f in zip(runs, got):
        with SodBatch([run], **kw) as b:
            b.step(21)
            np.testing.assert_array_equal(f, np.stack(list(b.moments(0).values())))
