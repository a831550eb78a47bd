"""The tiles of the temporally blocked 1D kernel in FP64 and the mixed mode (one tile an SM up to a number of cells an SM,
two of 128 cells or more beyond) against one launch per stage, at the edges of that rule and on the smallest grids."""
import numpy as np
import pytest

from paper_2403_13406_gb300 import eslbm, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

SMS = torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("n", [2, 9, 257, 8 * SMS + 1, 232 * SMS, 232 * SMS + 1, 248 * SMS, 248 * SMS + 1, 256 * SMS + 1])
@pytest.mark.parametrize("mode,precision", [("fixed", "fp64"), ("entropic", "fp64"), ("entropic", "fp32_mixed")])
def test_tiles_match_per_stage(n, mode, precision):
    """FP64 to 1e-13 relative (the same relaxation, contracted by the compiler in two kernels), mixed to the FP32 bar."""
    out = []
    for blocking in (True, False):
        sim = eslbm.Simulation(eslbm.make_config(1, "sw", n, 1, V=4.0, g=9.81, precision=precision, omega_mode=mode,
                                                 blocking=blocking))
        sim.init_equilibrium(inputs.sw_sine_1d(n, 1.0, 0.1))
        sim.step(2)
        out.append(sim.distributions(host=True))
        sim.close()
    if precision == "fp64":
        assert np.abs(out[0] - out[1]).max() <= 1e-13 * np.abs(out[1]).max()
    else:
        assert np.linalg.norm(out[0] - out[1]) <= 1e-5 * np.linalg.norm(out[1])
