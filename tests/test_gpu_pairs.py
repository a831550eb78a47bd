"""Init and read-back of FP32 lattices, which compute in pairs of FP32 numbers: the results are the FP32 rounding of
the FP64 equilibrium and the FP64 sum of the populations, over ordinary, zero, tiny, huge and non-finite values."""
import numpy as np
import pytest

import oracle as O
from paper_2403_13406_gb300 import eslbm, inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CASES = {
    "burgers1d": (1, "burgers", 1003, 1, dict(V=1.5)),
    "linear2d": (2, "linear", 61, 17, dict(V=1.0, a=(0.2, -0.15))),
    "burgers2d": (2, "burgers", 61, 17, dict(V=3.0, c=(1.0, 0.6))),
    "sw1d": (1, "sw", 1003, 1, dict(V=4.0, g=9.81)),
    "sw2d": (2, "sw", 61, 17, dict(V=8.0, g=9.81)),
    "euler2d": (2, "euler", 61, 17, dict(V=8.0, gamma=1.4)),
}


def fields(name):
    dim, system, nx, ny, kw = CASES[name]
    rng = np.random.default_rng(5)
    n = nx * ny
    if system in ("burgers", "linear"):
        u = rng.uniform(-1, 1, (1, n))
        u[0, :40] = 10.0 ** rng.uniform(-300, -5, 40)
        u[0, 40:50] = 0.0
    elif system == "sw":
        u = np.stack([1 + 0.3 * rng.uniform(-1, 1, n)] + [0.2 * rng.uniform(-1, 1, n) for _ in range(dim)])
        u[0, :20] = 10.0 ** rng.uniform(-20, -3, 20)
        u[1:, :20] = 0.0
        u[1:, 20:40] *= 1e-30
    else:
        rho, v, w, p = (rng.uniform(0.5, 1.5, n), rng.uniform(-1, 1, n), rng.uniform(-1, 1, n), rng.uniform(0.5, 1.5, n))
        u = np.stack([rho, rho * v, rho * w, 2.5 * p + 0.5 * rho * (v * v + w * w)])
        u[1, :20] = 0.0
        u[2, 10:30] *= 1e-25
        u[:, 30:40] *= 1e15
        u[3, 40:50] = 0.5 * (u[1] ** 2 + u[2] ** 2)[40:50] / u[0, 40:50] * (1 + 1e-9)  # almost no pressure
    return u.reshape((u.shape[0],) + ((nx,) if dim == 1 else (ny, nx)))


@pytest.mark.parametrize("name", list(CASES))
def test_init_is_the_rounded_equilibrium(name):
    """Each population is the FP64 one rounded to FP32 (at most one unit in the last place off where the
    FP64 value lies within its own rounding of a tie, or where opposite terms cancel)."""
    dim, system, nx, ny, kw = CASES[name]
    u = fields(name)
    ref = O.init_equilibrium(O.Model(dim, system, nx, ny, **kw), u)
    sim = eslbm.Simulation(eslbm.make_config(dim, system, nx, ny, precision="fp32", **kw))
    sim.init_equilibrium(torch.from_numpy(u).cuda())
    f = sim.distributions(host=True)
    sim.close()
    scale = np.abs(ref).reshape(ref.shape[0], -1).max(axis=0).reshape((1,) + ref.shape[1:])
    r32 = ref.astype(np.float32).astype(np.float64)
    assert (np.abs(f - r32) <= np.spacing(np.abs(r32).astype(np.float32)).astype(np.float64) + 2.0 ** -45 * scale).all()
    assert (f == r32).mean() > 0.999


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("shifted", [False, True])
def test_moments_are_the_fp64_sums(name, shifted):
    dim, system, nx, ny, kw = CASES[name]
    m = O.Model(dim, system, nx, ny, **kw)
    rng = np.random.default_rng(9)
    f0 = (rng.standard_normal((m.q * m.M,) + m.grid_shape) * 10.0 ** rng.uniform(-6, 6, m.grid_shape)).astype(np.float32).astype(np.float64)
    f0.reshape(m.q * m.M, -1)[:, :5] = 0.0
    f0.reshape(m.q * m.M, -1)[:, 5:8] = 3.2e38  # the FP32 sum overflows, the FP64 one does not
    uref = {"burgers": (0.5,), "linear": (0.5,), "sw": (1.0, 0.0, 0.0)[:m.M], "euler": (1.0, 0.0, 0.0, 2.5)}[system]
    sim = eslbm.Simulation(eslbm.make_config(dim, system, nx, ny, precision="fp32", u_ref=uref if shifted else None, **kw))
    sim.init_distributions(f0)
    f = sim.distributions(host=True).reshape((m.q, m.M) + m.grid_shape)
    u = sim.moments().cpu().numpy()
    sim.close()
    # shifted: the populations read back are the stored ones plus their reference, each rounded once
    bound = 4 * 2.0 ** -52 * np.abs(f).sum(axis=0) + (4 * 2.0 ** -52 if shifted else 0.0)
    assert (np.abs(u - f.sum(axis=0)) <= bound).all()


def test_domain_edge_and_non_finite_values():
    """Refused where the FP64 test refuses: just outside the domain, NaN and infinities; accepted just inside."""
    V = 1.5
    sim = eslbm.Simulation(eslbm.make_config(1, "burgers", 64, V=V, precision="fp32"))
    u = np.full((1, 64), 0.5)
    u[0, 7] = V * (1 - 1e-12)
    sim.init_equilibrium(u)
    for bad, status in ((V, eslbm.ERR_DOMAIN), (-V * (1 + 1e-12), eslbm.ERR_DOMAIN), (np.nan, eslbm.ERR_NAN), (np.inf, eslbm.ERR_NAN)):
        u[0, 7] = bad
        with pytest.raises(eslbm.EslbmError) as e:
            sim.init_equilibrium(u)
        assert e.value.status == status
    sim.close()
