"""Initialisation of FP32 lattices where the terms of a population cancel: u_m / q against phi / (2V), or the pressure's
two terms.  Every population is the FP32 rounding of its own value, however small it is against its terms."""
import numpy as np
import pytest

from paper_2403_13406_gb300 import eslbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

N, V, G, GAMMA = 20000, 8.0, 9.81, 1.4


def fields(system, dim):
    """States whose +x momentum population f = q_x / q - (q_x^2 / h + p) / (2V) of the opposite direction is 1e-2 ... 1e-9
    of its terms."""
    rng = np.random.default_rng(4)
    L = np.longdouble
    q = 2 * dim
    h = 0.3 + 0.2 * rng.uniform(0, 1, N)
    eps = rng.choice([-1, 1], N) * 10.0 ** rng.uniform(-9, -2, N)
    if system == "sw":
        p = G * h.astype(L) ** 2 / 2
    else:
        p = (0.2 + 0.1 * rng.uniform(0, 1, N)).astype(L)
    # q_x / q = (1 + eps) (q_x^2 / h + p) / (2V): the smaller root
    b = V * L(2) / q / (1 + eps)
    qx = h * (b - np.sqrt(b * b - 4 * p / h)) / 2
    rows = [h, qx.astype(np.float64)] + [0.1 * h * rng.uniform(-1, 1, N)] * (dim - 1)
    if system == "euler":
        rows.append((p / (GAMMA - 1) + (qx ** 2 + L(1) * rows[2] ** 2) / h / 2).astype(np.float64))
    return np.stack(rows)


def equilibrium(system, dim, u):
    L = np.longdouble
    u = u.astype(L)
    p = L(G) * u[0] ** 2 / 2 if system == "sw" else L(GAMMA - 1.0) * (u[3] - (u[1] ** 2 + u[2] ** 2) / u[0] / 2)
    d = []
    for j in range(dim):
        v = u[1 + j] / u[0]
        f = [u[1 + j]] + [u[1 + i] * v + (p if i == j else 0) for i in range(dim)]
        d.append(np.stack(f + ([v * (u[3] + p)] if system == "euler" else [])) / (2 * L(V)))
    base = u / (2 * dim)
    terms = np.stack([np.abs(base) + np.abs(x) for x in d] * 2)
    return np.stack([base + x for x in d] + [base - x for x in d]), terms


@pytest.mark.parametrize("shifted", [False, True])
@pytest.mark.parametrize("system,dim", [("sw", 1), ("sw", 2), ("euler", 2)])
def test_populations_left_of_cancelling_terms(system, dim, shifted):
    """Bound: the rounding to FP32 (2^-24 of the value, a hundredth more) and eight roundings of the terms in 64 bits."""
    u = fields(system, dim)
    uref = {"sw": (0.4, 0.1, 0.0)[:1 + dim], "euler": (0.4, 0.1, 0.0, 0.7)}[system] if shifted else None
    kw = dict(V=V, g=G) if system == "sw" else dict(V=V, gamma=GAMMA)
    sim = eslbm.Simulation(eslbm.make_config(dim, system, N, 1, precision="fp32", u_ref=uref, **kw))
    sim.init_equilibrium(torch.from_numpy(u).cuda())
    stored = sim._fa.view(torch.float32)[:sim.planes * N].cpu().numpy().astype(np.longdouble).reshape(2 * dim, 1 + dim + (system == "euler"), N)
    sim.close()
    feq, terms = equilibrium(system, dim, u)
    if shifted:  # subtract the reference as it is stored: the populations of a lattice at u_ref, read back plus fbar
        sim = eslbm.Simulation(eslbm.make_config(dim, system, N, 1, precision="fp32", u_ref=uref, **kw))
        sim.init_distributions(np.zeros((sim.planes,) + sim.grid_shape))
        fbar = -sim._fa.view(torch.float32)[:sim.planes * N].cpu().numpy().astype(np.longdouble).reshape(stored.shape)
        sim.close()
        feq = feq - fbar
        terms = terms + np.abs(fbar)
    assert (np.abs(stored - feq) <= 1.01 * 2.0 ** -24 * np.abs(feq) + 8 * 2.0 ** -53 * terms).all()
    if not shifted:  # the values are what the test says it looks at
        assert (np.abs(feq) < 1e-7 * terms).any()
