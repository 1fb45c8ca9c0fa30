"""FP32 grids of up to 640 000 nodes take a kernel that updates one 64 x 4 tile per
CTA without a march.  Its arithmetic is the march's: the same flow repeated in y
(periodic) past that size gives the same bits, at tile edges and on grids
smaller than the stencil, also after the equilibrium shift has moved.
"""
import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=4.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=20.0, rho_v=1.0, nu_l=0.6, nu_v=0.1,
           Gx=1e-6, Gy=-2e-6)
MOST = 640000


@pytest.mark.parametrize("shape", [(64, 4), (65, 5), (63, 3), (1, 1), (3, 7), (130, 9), (66, 6)])
def test_shot_equals_march(oracle_mod, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    nx, ny = shape
    times = MOST // (nx * ny) + 1
    o = oracle_mod.Oracle(shape, **PRM)
    o.init_phi(wl.droplet(nx, ny, 0.3 * min(nx, ny) + 1.0, 4.0))
    f, g, S = o.get_state()
    g = g + wl.perturbed_state(g.shape, 1e-3, 15)
    S = S + wl.perturbed_state(S.shape, 1e-4, 16)
    a = sim.Simulation(shape, precision="fp32", **PRM)
    b = sim.Simulation((nx, ny * times), precision="fp32", **PRM)
    rep = lambda v: np.concatenate([v.reshape(-1, ny, nx)] * times, axis=1)  # noqa: E731
    a.set_state(f, g, S, 0)
    b.set_state(rep(f), rep(g), rep(S), 0)
    o.set_state(*a.get_state(), 0)
    a.step(1)
    b.step(1)
    o.step(1)
    ma, mo = a.moments(), o.macros()
    assert np.abs(ma["phi"] - mo["phi"]).max() <= 1e-5
    assert np.abs(ma["u"] - mo["u"]).max() <= 1e-6
    da, db = a.diagnostics(), b.diagnostics()  # move both shifts to the middle of the mu range
    assert da["mu_min"] == db["mu_min"] and da["mu_max"] == db["mu_max"]
    a.step(4)
    b.step(4)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x.reshape(-1, ny, nx), y.reshape(-1, ny * times, nx)[:, :ny])
        assert np.array_equal(x.reshape(-1, ny, nx), y.reshape(-1, ny * times, nx)[:, -ny:])
    a.close()
    b.close()
