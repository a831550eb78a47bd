"""The entropic omega of fields at the ends of the floating-point range.

The coefficient c_2 of the expansion of the entropy scales with the square of the fields, so in thin films it is
subnormal (or zero) while depth, velocity and deviations are ordinary numbers.  Cells a little off equilibrium have
omega = 2 up to a few times their relative deviation, whatever the depth.
"""
import numpy as np
import pytest

from paper_2403_13406_gb300 import eslbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

N, G = 4096, 9.81


def equilibrium(dim, u, V):
    """f^eq_k = u / q + sign_k phi^j(u) / (2V) in extended precision, q_i q_j / h as q_i (q_j / h): the oracle's product
    of two momenta leaves the range of doubles at these depths."""
    u = u.astype(np.longdouble)
    q = 2 * dim
    feq = np.empty((q,) + u.shape, dtype=np.longdouble)
    for j in range(dim):
        phi = np.stack([u[1 + j]] + [u[1 + i] * (u[1 + j] / u[0]) for i in range(dim)])
        phi[1 + j] += G * u[0] * u[0] / 2
        feq[j] = u / q + phi / (2 * V)
        feq[j + dim] = u / q - phi / (2 * V)
    return feq


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("precision,depths", [
    ("fp32", (1e-15, 1e-18, 1e-21, 1e-24, 1e-27, 1e-30, 1e-33)),
    ("fp32_mixed", (1e-18, 1e-24, 1e-30)),
    ("fp64", (1e-200, 1e-290, 1e-293, 1e-296, 1e-299, 1e-302)),
])
def test_thin_films_relax_with_omega_near_two(dim, precision, depths):
    """Moving films (|v| <= 0.3) with deviations of 1e-7 ... 1e-5 of the populations: |omega - 2| <= 0.01 per cell.
    The bound adds sixteen roundings of the cell's largest value and a few steps of the subnormal numbers."""
    V = 4.0 if dim == 1 else 8.0
    ulp, tiny = (2.0 ** -53, 2.0 ** -1074) if precision == "fp64" else (2.0 ** -24, 2.0 ** -149)
    for h in depths:
        rng = np.random.default_rng(5)
        q, M = 2 * dim, 1 + dim
        u = np.zeros((M, N))
        u[0] = h * (1 + 0.2 * rng.uniform(-1, 1, N))
        for j in range(dim):
            u[1 + j] = u[0] * 0.3 * rng.uniform(-1, 1, N)
        d = rng.uniform(-1, 1, (q, M, N)) * 10.0 ** rng.uniform(-7, -5, N)
        d[:, 1:] *= V / 2
        d -= d.mean(axis=0)
        f = (equilibrium(dim, u, V) + u[0] * d / q).astype(np.float64)
        if precision != "fp64":
            f = f.astype(np.float32).astype(np.float64)
        delta = equilibrium(dim, f.astype(np.longdouble).sum(axis=0), V) - f

        sim = eslbm.Simulation(eslbm.make_config(dim, "sw", N, 1, precision=precision, omega_mode="entropic", V=V, g=G))
        sim.init_distributions(f)
        sim.relax()
        out, fallbacks = sim.distributions(host=True).reshape(f.shape), sim.diagnostics()["fallbacks"]
        sim.close()

        cellmax = lambda a: np.abs(a).max(axis=(0, 1))
        assert np.isfinite(out).all(), h
        assert fallbacks == 0, h
        assert (cellmax(out - (f + 2 * delta)) <= 0.01 * cellmax(delta) + 16 * ulp * cellmax(f) + 16 * tiny).all(), h
