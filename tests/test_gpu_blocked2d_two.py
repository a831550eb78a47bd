"""FP32 Euler through the temporally blocked 2D kernel two stages a launch (its default) against one launch per stage.

Plain storage takes the kernel's form with one item a consumer, whose relaxation leaves nothing to the compiler:
the two paths agree to the last bit.  Shifted storage takes the general form, whose contractions may differ.  Sizes: one
strip and segment, several of both with short last ones, windows wider than the grid.
"""
import numpy as np
import pytest

from paper_2403_13406_gb300 import eslbm, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def run(nx, ny, scheme, shifted, blocking):
    cfg = eslbm.make_config(2, "euler", nx, ny, V=8.0, gamma=1.4, precision="fp32", omega_mode="fixed", scheme=scheme,
                            blocking=blocking, u_ref=(1.0, 1.0, 1.0, 3.5) if shifted else None)
    sim = eslbm.Simulation(cfg)
    sim.init_equilibrium(inputs.euler_vortex_2d(nx, ny))
    sim.step(2)
    f = sim.distributions(host=True)
    sim.close()
    return f


# 508 and 764 columns: three and four strips of at most 248 (240 for the group of shifts -1 and -4), the last one short;
# 300 and 77 rows: several segments of 32 rows or more, the last one short
@pytest.mark.parametrize("nx,ny", [(8, 6), (40, 36), (248, 33), (252, 65), (416, 300), (508, 300), (764, 77)])
@pytest.mark.parametrize("scheme", ["I", "III"])
@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("blocking", [True, 2])
def test_two_stages_a_launch(nx, ny, scheme, shifted, blocking):
    a, b = run(nx, ny, scheme, shifted, blocking), run(nx, ny, scheme, shifted, False)
    if shifted:
        assert np.abs(a - b).max() <= 1e-6 * np.abs(b).max()
    else:
        assert np.array_equal(a, b)
