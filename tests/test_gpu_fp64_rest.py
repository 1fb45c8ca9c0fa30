"""The FP64 rest population, which is nearly phi, is rounded once per step.

Its change in a step is small beside it, so the change is formed first and added:
forming the sum term by term rounds at the size of phi three times, and phi
then loses accuracy 1.7 times as fast.  A uniform flow at rest with S_prev of the last
step varying from node to node has the exact new value
f_0 + (s - (1 - w_0) alpha mu)/tau_f - w_0 b_0 S_prev/2, s the sum of the moving populations: the
result is off by half an ulp and a few roundings of the small terms.
"""
from fractions import Fraction as Fr

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PRM = dict(W=4.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=10.0, rho_v=1.0, nu_l=0.1, nu_v=0.1)


@pytest.mark.parametrize("name,shape", [("D2Q9", (16, 128)), ("D2Q9", (130, 64)),
                                        ("D3Q19", (33, 10, 9))])
def test_rest_population_is_rounded_once(name, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    N = int(np.prod(shape))
    w0, b0, w = ((Fr(4, 9), -2, [1 / 9] * 4 + [1 / 36] * 4) if name == "D2Q9" else
                 (Fr(1, 3), Fr(-5, 2), [1 / 18] * 6 + [1 / 36] * 12))
    rng = np.random.default_rng(9)
    f = np.empty((len(w) + 1, N))
    f[0] = 0.7310585786300049
    f[1:] = 1.3e-3 * np.array(w)[:, None]
    S = 1e-3 * rng.uniform(-1.0, 1.0, N)
    s = sim.Simulation(shape, lattice=name, precision="fp64", **PRM)
    s.set_state(f, np.zeros_like(f), S, 0)
    s.step(1)
    got = s.get_state()[0][0].ravel()
    moving = sum(Fr(x) for x in f[1:, 0])
    phi = Fr(f[0, 0]) + moving
    mu = 4 * Fr(s.beta) * (phi - 1) * phi * (phi - Fr(1, 2))
    itf = 1 / Fr(s.tau_f)
    change = itf * (moving - (1 - w0) * Fr(s.alpha) * mu)
    small = float(itf * (moving + abs(mu))) + np.abs(S).max()
    tol = Fr(0.5 * np.spacing(1.0) / 2 + 8.0 * 2.0 ** -53 * small)  # ulp of [1/2, 1)
    assert got.min() > 0.5 and got.max() < 1.0
    worst = max(abs(Fr(g) - (Fr(f[0, 0]) + change - w0 * b0 * Fr(p) / 2))
                for g, p in zip(got.tolist(), S.tolist()))
    assert worst <= tol, float(worst / tol)
    s.close()
