"""The FP64 collisions keep phi and momentum for any relaxation time.

A population relaxes as f + (f^eq - f)/tau, and its moments stay because every
population is moved by the same 1/tau.  The form f (1 - 1/tau) + f^eq/tau moves it
by 1 - fl(1 - 1/tau): for tau > 2 that differs from 1/tau by up to 2^-54, and the sums
then drift by that much of themselves in every step.  The tests take a tau at which it
differs most and a flow whose exact moments stay (no surface tension, no
force), and bound the drift by what independent roundings give: 8 sqrt(nodes x
steps) of the largest population's rounding, and for the momentum also 8
roundings of its relaxed part per step.  The drift of the second form is tens of
times that.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
STEPS = 400
CASES = [("D2Q9", (16, 128)), ("D2Q9", (130, 64)), ("D3Q19", (34, 10, 9))]


def lattice(name):
    if name == "D2Q9":
        c = [(0, 0), (0, -1), (1, 0), (0, 1), (-1, 0), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    else:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
        for a, b in ((0, 1), (0, 2), (1, 2)):
            for s in ((1, 1), (1, -1), (-1, 1), (-1, -1)):
                v = [0, 0, 0]
                v[a], v[b] = s
                c.append(tuple(v))
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    return np.array(c, dtype=float), np.array(w)


def residue(rate):
    """What 1 - fl(1 - rate) exceeds rate by (exact for rate < 1/2)."""
    return (1.0 - (1.0 - rate)) - rate


def simulation(name, shape, **prm):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    return sim.Simulation(shape, lattice=name, precision="fp64", sigma=0.0, W=4.0, M=0.05,
                          rho_l=1.0, rho_v=1.0, **prm)


@pytest.mark.parametrize("name,shape", CASES)
def test_phi_of_a_slow_relaxation(name, shape):
    tau = max((300.0 + 0.25 * k for k in range(80)), key=lambda t: abs(residue(1.0 / t)))
    c, w = lattice(name)
    N = int(np.prod(shape))
    rng = np.random.default_rng(3)
    f = w[:, None] * rng.uniform(0.5, 1.5, (w.size, N))
    s = simulation(name, shape, tau_f=tau, nu_l=0.1, nu_v=0.1)
    s.set_state(f, np.zeros_like(f), np.zeros(N), 0)
    s.step(STEPS)
    g = s.get_state()[0].reshape(w.size, N)
    bound = 8.0 * math.sqrt(N * STEPS) * EPS * f.max()
    # the drift the other form would have: most of the moving part is still there
    assert abs(residue(1.0 / tau)) * 0.25 * f[1:].sum() * STEPS > 10.0 * bound
    assert not np.array_equal(g, f)
    assert abs(math.fsum(g.ravel()) - math.fsum(f.ravel())) <= bound
    s.close()


@pytest.mark.parametrize("name,shape", CASES)
def test_momentum_of_a_slow_relaxation(name, shape):
    nu = max((333.0 + 0.25 * k for k in range(80)), key=lambda v: abs(residue(1.0 / (3.0 * v + 0.5))))
    c, w = lattice(name)
    N = int(np.prod(shape))
    rng = np.random.default_rng(4)
    u = np.array([0.05, -0.03, 0.04])[:c.shape[1]]
    g = 3.0 * w[:, None] * (c @ u)[:, None] + 1e-3 * rng.uniform(-1.0, 1.0, (w.size, N))
    f = np.zeros_like(g)
    f[0] = 1.0
    s = simulation(name, shape, tau_f=1.0, nu_l=nu, nu_v=nu)
    s.set_state(f, g, np.zeros(N), 0)
    s.step(STEPS)
    h = s.get_state()[1].reshape(w.size, N)
    rate = 1.0 / (3.0 * nu + 0.5)
    assert not np.array_equal(h, g)
    for d in range(c.shape[1]):
        p0, p1 = (math.fsum((c[:, d:d + 1] * x).ravel()) for x in (g, h))
        bound = (8.0 * math.sqrt(N * STEPS) * EPS * np.abs(g).max() +
                 8.0 * EPS * rate * abs(p0) * STEPS)
        assert abs(residue(rate)) * abs(p0) * STEPS > 5.0 * bound
        assert abs(p1 - p0) <= bound
    s.close()
