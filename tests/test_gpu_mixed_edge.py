"""FP32_MIXED next to the edge of the convexity domain: no relaxation increases the cell's microscopic entropy.

Cells with |v| + sqrt(g h) up to the domain's bound 2V/q and deviations of 1e-7 ... 0.5 of the populations, where the
root of F(t) = B(t) - B(-1) is sensitive to every constant of B.  Cells without a root (or that leave the domain) fall
back to omega = 1 and are counted as such; the check of all others is the diagnostics' own, to 64 roundings of FP64.
"""
import numpy as np
import pytest

import oracle as O
from paper_2403_13406_gb300 import eslbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

N, G = 1 << 18, 9.81


# (V = 4 and 8: 1 / (2V) is a power of two; 3.7 and 7.3: it is rounded)
@pytest.mark.parametrize("dim,V", [(1, 4.0), (1, 3.7), (2, 8.0), (2, 7.3)])
def test_no_entropy_increase_next_to_the_edge(dim, V):
    rng = np.random.default_rng(11)
    m = O.Model(dim, "sw", N, 1, V=V, g=G)
    nu = 2 * V / m.q
    u = np.zeros((m.M, N))
    u[0] = rng.uniform(0.4, 0.9999 * nu ** 2 / G, N)
    for j in range(dim):
        u[1 + j] = u[0] * (nu - np.sqrt(G * u[0])) * 0.999 * rng.uniform(-1, 1, N)
    f = O.init_equilibrium(m, u.reshape((m.M,) + m.grid_shape)).reshape(m.q, m.M, N)
    d = rng.uniform(-1, 1, f.shape) * 10.0 ** rng.uniform(-7, -0.3, N)
    d[:, 1:] *= V / 2
    d -= d.mean(axis=0)
    f = f + u[0] * d / m.q
    sim = eslbm.Simulation(eslbm.make_config(dim, "sw", N, 1, precision="fp32_mixed", omega_mode="entropic", V=V, g=G,
                                             diagnostics=True))
    sim.init_distributions(np.ascontiguousarray(f.reshape((m.q * m.M,) + m.grid_shape)))
    sim.relax()
    diag = sim.diagnostics()
    sim.close()
    assert diag["fallbacks"] < N // 2
    assert diag["entropy_increases"] == 0, diag
    assert diag["entropy_excess_max"] <= 64 * 2.220446e-16
