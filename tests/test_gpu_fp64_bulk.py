"""The chemical potential of the FP64 D2Q9 step in and near the bulk phases.

psi'(phi) = 4 beta (phi - phi_l)(phi - phi_v)(phi - phibar) vanishes at both phases.  Formed
from these factors it is exactly zero there and accurate to a few roundings
beside them, whatever the phases' values; formed as t (t^2 - (dphi/2)^2) with
t = phi - phibar it keeps the rounding of t^2, an error that does not shrink with
the distance from the phase.  Both FP64 step kernels: 16 x 8 nodes (the update of
a small grid, split over four warps) and 200 x 130 (the tile march).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PRM = dict(W=4.0, M=0.05, alpha=1.0, sigma=1e-2, phi_l=1.2, phi_v=0.1, rho_l=20.0, rho_v=1.0,
           nu_l=0.1, nu_v=0.1)
SHAPES = [(16, 8), (200, 130)]
W = np.array([4.0] + [1.0] * 4 + [0.25] * 4) / 9.0


def simulation(shape, phi):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    s = sim.Simulation(shape, precision="fp64", **PRM)
    s.init_phi(np.full(shape[::-1], phi))
    return s


@pytest.mark.parametrize("phi", [PRM["phi_l"], PRM["phi_v"]])
@pytest.mark.parametrize("shape", SHAPES)
def test_a_uniform_bulk_phase_is_exactly_at_rest(shape, phi):
    s = simulation(shape, phi)
    s.step(3)
    m = s.moments()
    f, g, S = s.get_state()
    assert np.all(m["phi"] == phi) and np.all(m["mu"] == 0.0) and np.all(m["u"] == 0.0)
    assert np.all(f[0] == phi) and np.all(f[1:] == 0.0)
    assert np.all(g == 0.0) and np.all(S == 0.0)
    s.close()


@pytest.mark.parametrize("d", [1e-9, -3e-10, 1e-13])
@pytest.mark.parametrize("phase", ["phi_l", "phi_v"])
@pytest.mark.parametrize("shape", SHAPES)
def test_mu_beside_a_phase_to_a_few_roundings(shape, phase, d):
    """phi - phase is exact, and five more operations round: 1e-14 covers them
    (and the relaxation's four, amplified by |1 - 1/tau_f| + 1/tau_f = 2.1)."""
    s = simulation(shape, PRM[phase] + d)
    m = s.moments()
    f0 = s.get_state()[0]
    phi, mu = m["phi"].flat[0], m["mu"].flat[0]
    pb = 0.5 * (PRM["phi_l"] + PRM["phi_v"])
    ref = 4.0 * s.beta * (phi - PRM["phi_l"]) * (phi - PRM["phi_v"]) * (phi - pb)
    assert ref != 0.0 and np.all(m["phi"] == phi)
    assert abs(mu - ref) <= 1e-14 * abs(ref)
    s.step(1)
    f = s.get_state()[0]
    itf = 1.0 / s.tau_f
    for i in range(1, 9):
        want = (1.0 - itf) * f0[i].flat[0] + W[i] * itf * s.alpha * ref
        assert np.abs(f[i] - want).max() <= 1e-14 * abs(want)
    s.close()
