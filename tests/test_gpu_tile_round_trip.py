"""The tile width that rslb_launch_info reports can be asked for and gives bitwise the
automatic choice's populations."""
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


@pytest.mark.parametrize("precision,Z,Q_xi", [
    ("f64", 7, 8), ("f64", 200, 20), ("f64", 500, 20), ("f64", 900, 50), ("f64", 3000, 20),
    ("f64", 70, 300), ("f32", 300, 8), ("f32", 300, 20), ("f32", 300, 50), ("f32", 40, 333)])
def test_reported_tile_is_accepted(precision, Z, Q_xi):
    from paper_1612_01287_gb300 import Sod
    kw = dict(Z=Z, Q_xi=Q_xi, Q_L=3, precision=precision, tau=5e-3, dt=min(1e-3, 0.5 / Z))
    out, tile = [], 0
    for _ in range(2):
        with Sod(tile_cells=tile, **kw) as s:
            s.step(4)
            tile = s.launch_info()[0]
            out.append((tile, s.get_state()))
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])
