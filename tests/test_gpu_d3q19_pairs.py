"""The FP32 D3Q19 pass updates two x-neighbours per thread, with 64-bit loads and
stores of both where rows have an even number of nodes and single values where
they do not.  Both forms do the same arithmetic: a grid of odd width and the
same grid repeated twice in x (periodic: the same flow) give the same bits, at
widths around the 32-node tile; and one step agrees with the oracle within the
FP32 bounds (phi 1e-5, u 1e-6 absolute).
"""
import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=5.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=10.0, rho_v=1.0, nu_l=1.0, nu_v=0.1,
           Gx=1e-6, Gy=-2e-6, Gz=5e-7)


def twice(a, nx):
    a = a.reshape(-1, nx)
    return np.ascontiguousarray(np.concatenate([a, a], axis=1))


@pytest.mark.parametrize("shape", [(1, 5, 3), (31, 8, 4), (33, 9, 5), (17, 1, 7), (65, 10, 2),
                                   (35, 3, 1)])
def test_odd_rows_equal_repeated_even_rows(oracle_mod, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    nx, ny, nz = shape
    o = oracle_mod.Oracle(shape, lattice_name="D3Q19", **PRM)
    o.init_phi(wl.two_droplets(nx, ny, min(shape) / 4 + 1.0, 5.0, nz=nz))
    f, g, S = o.get_state()
    g = g + wl.perturbed_state(g.shape, 1e-3, 31)
    S = S + wl.perturbed_state(S.shape, 1e-4, 32)
    a = sim.Simulation(shape, lattice="D3Q19", precision="fp32", diag_every=2, **PRM)
    b = sim.Simulation((2 * nx, ny, nz), lattice="D3Q19", precision="fp32", diag_every=2, **PRM)
    a.set_state(f, g, S, 0)
    b.set_state(twice(f, nx), twice(g, nx), twice(S, nx), 0)
    o.set_state(*a.get_state(), 0)
    a.step(1)
    o.step(1)
    ma, mo = a.moments(), o.macros()
    assert np.abs(ma["phi"] - mo["phi"]).max() <= 1e-5
    assert np.abs(ma["u"] - mo["u"]).max() <= 1e-6
    a.diagnostics()  # moves the equilibrium shift: the next step writes with another one
    b.step(1)
    b.diagnostics()
    a.step(3)
    b.step(3)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(twice(x, nx).ravel(), y.ravel())
    ma, mb = a.moments(), b.moments()
    for k in ma:
        assert np.array_equal(twice(ma[k], nx).ravel(), mb[k].ravel())
    da, db = a.last_diagnostics(), b.last_diagnostics()
    assert da["u_max"] == db["u_max"] and da["mu_max"] == db["mu_max"]
    assert np.isclose(2 * da["sum_phi"], db["sum_phi"], rtol=1e-12)
    a.close()
    b.close()
