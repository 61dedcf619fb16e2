"""The WENO weights do not see a factor of f: populations scaled by a power of two
stay the scaled trajectory as far as the squares of their differences are normal
FP64 numbers."""
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


def _run(k, mode, Z, Q_xi, tile):
    from paper_1612_01287_gb300 import Sod
    z = (np.arange(Z) + 0.5) / Z
    fields = (1.0 + 0.3 * np.sin(7 * z) + (z > 0.6), 1.0 + 0.2 * np.cos(5 * z),
              0.5 * np.sin(9 * z + 1))
    with Sod(Z=Z, Q_xi=Q_xi, Q_L=3, precision="f64", bc="outflow", tau_mode=mode, tau=5e-3,
             dt=1e-3, fields=fields, tile_cells=tile) as s:
        s.set_state(s.get_state() * 2.0 ** k)
        s.step(10)
        return s.get_state() * 2.0 ** -k


@pytest.mark.parametrize("mode,k", [("none", k) for k in (-300, -370, -384, -400, -480, 400)] +
                         [("const", k) for k in (-370, -384, -400, 400)])
@pytest.mark.parametrize("Z,Q_xi,tile", [(60, 20, 0), (60, 20, 16), (60, 200, 8)])
def test_scaled_populations_follow_the_scaled_trajectory(mode, k, Z, Q_xi, tile):
    """Every operation commutes with the factor 2^k; only squares that underflow (at
    2^-480 those of differences below ~1e-9 of f, far below the ones here) do not."""
    ref = _run(0, mode, Z, Q_xi, tile)
    assert np.abs(_run(k, mode, Z, Q_xi, tile) - ref).max() <= 1e-13 * np.abs(ref).max()
