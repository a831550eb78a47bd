"""The entropic omega from the expansion of the entropy about the equilibrium, against the oracle's dichotomy.

One relaxation of cells whose distance from equilibrium sweeps the ranges of the three routes: rounding level
(omega = 2), the truncated expansion, Newton on the closed form, and the general search (near the edge of
the convexity domain), with bounds of the search interval on both sides of the root.
"""
import numpy as np
import pytest

import oracle as O
from paper_2403_13406_gb300 import eslbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

N = 3000
SYSTEMS = {
    "burgers1d": (1, "burgers", dict(V=1.5)),
    "burgers2d": (2, "burgers", dict(V=3.0, c=(1.0, 0.6))),
    "sw1d": (1, "sw", dict(V=4.0, g=9.81)),
    "sw2d": (2, "sw", dict(V=8.0, g=9.81)),
}


def cells(dim, system, kw, most, fp32):
    """Equilibria plus deviations of relative size 1e-12 ... most (log-uniform), summing to zero per component;
    every eleventh cell is at equilibrium."""
    rng = np.random.default_rng(77)
    m = O.Model(dim, system, N, 1, **kw)
    u = np.zeros((m.M, N))
    if system == "burgers":
        u[0] = 0.5 + 0.4 * rng.uniform(-1, 1, N)
    else:
        u[0] = 1.0 + 0.3 * rng.uniform(-1, 1, N)
        for j in range(dim):
            u[1 + j] = u[0] * 0.2 * rng.uniform(-1, 1, N)
    f = O.init_equilibrium(m, u.reshape((m.M,) + m.grid_shape)).reshape(m.q, m.M, N)
    d = rng.uniform(-1, 1, f.shape) * 10.0 ** rng.uniform(-12, np.log10(most), N)
    d[:, 1:] *= kw["V"] / 2
    d -= d.mean(axis=0)
    d[:, :, ::11] = 0.0
    f = f + d / m.q
    if fp32:
        f = f.astype(np.float32).astype(np.float64)
    return np.ascontiguousarray(f.reshape((m.q * m.M,) + m.grid_shape))


def relaxed(dim, system, kw, f, precision, t_max):
    sim = eslbm.Simulation(eslbm.make_config(dim, system, N, 1, precision=precision, omega_mode="entropic", t_max=t_max, **kw))
    sim.init_distributions(f)
    sim.relax()
    out, fallbacks = sim.distributions(host=True), sim.diagnostics()["fallbacks"]
    sim.close()
    m = O.Model(dim, system, N, 1, omega_mode="entropic", t_max=t_max, **kw)
    ref, st = f.copy(), O.Stats()
    O.relax(m, ref, stats=st)
    return out, ref, fallbacks, st.fallbacks


@pytest.mark.parametrize("t_max", [3.0, 1.0005, 0.8])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_fp64(name, t_max):
    dim, system, kw = SYSTEMS[name]
    out, ref, fb, fb_ref = relaxed(dim, system, kw, cells(dim, system, kw, 0.3, False), "fp64", t_max)
    # with t_max below every root all cells but those at equilibrium fall back, and which of the cells are at
    # equilibrium (E0 = 0) is a matter of rounding
    if t_max > 1.0:
        assert fb == fb_ref
    assert np.abs(out - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("precision", ["fp32", "fp32_mixed"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_fp32(name, precision):
    """Per cell: sixteen roundings of the largest value (the moments, the equilibrium and the update) and an
    error of 1e-5 in omega times the deviation."""
    dim, system, kw = SYSTEMS[name]
    f = cells(dim, system, kw, 0.2, True)
    out, ref, fb, fb_ref = relaxed(dim, system, kw, f, precision, 3.0)
    assert fb == fb_ref
    scale = np.abs(f).reshape(f.shape[0], -1).max(axis=0)
    moved = np.abs(ref - f).reshape(f.shape[0], -1).max(axis=0)
    err = np.abs(out - ref).reshape(f.shape[0], -1).max(axis=0)
    assert (err <= 16 * 2.0 ** -24 * scale + 1e-5 * moved).all()
