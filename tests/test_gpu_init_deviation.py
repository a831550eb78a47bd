"""Initialisation of the shifted FP32 storage from small deviations: the stored values are the FP32 rounding of
f^eq(u) - fbar, relative to the deviation and not to f^eq."""
import numpy as np
import pytest

from paper_2403_13406_gb300 import eslbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CASES = {
    # dim, system, nx, ny, parameters, u_ref
    "linear1d": (1, "linear", 4001, 1, dict(V=1.0, a=(0.37, 0.0)), (0.75,)),
    "burgers1d": (1, "burgers", 4001, 1, dict(V=1.5), (0.5,)),
    "burgers2d": (2, "burgers", 77, 53, dict(V=3.0, c=(1.0, 0.6)), (0.5,)),
    "sw1d": (1, "sw", 4001, 1, dict(V=4.0, g=9.81), (1.0, 0.0)),
    "sw1d_moving": (1, "sw", 4001, 1, dict(V=3.7, g=9.81), (0.8, 0.15)),
    "sw2d": (2, "sw", 77, 53, dict(V=8.0, g=9.81), (1.0, 0.02, -0.01)),
    "euler2d": (2, "euler", 77, 53, dict(V=8.0, gamma=1.4), (1.0, 0.9, -0.4, 3.5)),
}


def equilibrium(dim, system, u, real, V=1.0, a=(0.0, 0.0), c=(1.0, 1.0), g=0.0, gamma=0.0):
    """f^eq_k,m = u_m / q + sign_k phi^j_m(u) / (2V) in extended precision, with the constants 1 / (2V), gamma - 1, ...
    rounded to the type `real`."""
    L = lambda x: np.longdouble(real(x))
    u = u.astype(np.longdouble)
    if system == "linear":
        phi = [np.stack([L(a[j]) * u[0]]) for j in range(dim)]
    elif system == "burgers":
        phi = [np.stack([L(c[j]) * u[0] * u[0] / 2]) for j in range(dim)]
    else:
        p = L(g) * u[0] ** 2 / 2 if system == "sw" else L(gamma - 1) * (u[3] - (u[1] ** 2 + u[2] ** 2) / u[0] / 2)
        phi = []
        for j in range(dim):
            v = u[1 + j] / u[0]
            f = [u[1 + j]] + [u[1 + i] * v + (p if i == j else 0) for i in range(dim)]
            phi.append(np.stack(f + ([v * (u[3] + p)] if system == "euler" else [])))
    q = 2 * dim
    d = [phi[j] * L(0.5 / V) for j in range(dim)]
    return np.stack([u / q + x for x in d] + [u / q - x for x in d])


@pytest.mark.parametrize("amplitude", [1e-2, 1e-4, 1e-6, 1e-8, 1e-9, 1e-10])
@pytest.mark.parametrize("name", list(CASES))
def test_stored_deviation(name, amplitude):
    """Bound: the rounding to FP32 (2^-24 of the value, a hundredth more for the pairs), the pairs' own 2^-43 of the
    cell's largest deviation, and eight roundings of f in 64 bits: four for the reference's own value (a constant of
    the lattice) and four for cells that are initialised in FP64 throughout."""
    dim, system, nx, ny, kw, uref = CASES[name]
    rng = np.random.default_rng(3)
    ref = np.array(uref).reshape(-1, 1)
    u = ref + amplitude * rng.uniform(-1, 1, (ref.shape[0], nx * ny))
    sim = eslbm.Simulation(eslbm.make_config(dim, system, nx, ny, precision="fp32", u_ref=uref, **kw))
    sim.init_equilibrium(torch.from_numpy(u).cuda())
    stored = sim._fa.view(torch.float32)[:sim.planes * nx * ny].cpu().numpy().astype(np.longdouble).reshape(-1, nx * ny)
    sim.close()
    feq = equilibrium(dim, system, u, np.float64, **kw).reshape(-1, nx * ny)
    # fbar: the equilibrium of u_ref with the constants of the storage precision's kernels, rounded to it
    fbar = equilibrium(dim, system, ref, np.float32, **kw).reshape(-1, 1)
    fbar = fbar.astype(np.float64).astype(np.float32).astype(np.longdouble)
    want = feq - fbar
    bound = 1.01 * 2.0 ** -24 * np.abs(want) + 2.0 ** -43 * np.abs(want).max(axis=0) + 8 * 2.0 ** -53 * np.abs(feq)
    assert (np.abs(stored - want) <= bound).all()
