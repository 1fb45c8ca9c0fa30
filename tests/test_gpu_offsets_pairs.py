"""The offset-storage pass updates two x-neighbours per thread, with 32-bit
loads and stores of both, where rows have an even number of nodes, and one node
per thread where they do not.  Both forms do the same arithmetic, so a grid of odd
width and the same grid repeated twice in x (periodic: the same flow) give the
same bits, at widths around the 32-node tile; and both agree with the oracle.
"""
import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=5.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=10.0, rho_v=1.0, nu_l=1.0, nu_v=0.1,
           Gx=1e-6, Gy=-2e-6, Gz=5e-7)
EPS = {"f16off": 2.0 ** -11, "bf16off": 2.0 ** -8}
SHAPES = [(1, 5, 3), (31, 8, 4), (33, 9, 5), (17, 1, 7), (65, 10, 2), (35, 3, 1)]


def start(oracle_mod, shape):
    nx, ny, nz = shape
    o = oracle_mod.Oracle(shape, lattice_name="D3Q19", **PRM)
    o.init_phi(wl.two_droplets(nx, ny, min(shape) / 4 + 1.0, 5.0, nz=nz))
    f, g, S = o.get_state()
    g = g + wl.perturbed_state(g.shape, 1e-3, 21)
    f = f + wl.perturbed_state(f.shape, 1e-4, 22)
    S = S + wl.perturbed_state(S.shape, 1e-4, 23)
    return o, f, g, S


def twice(a, nx):
    """The field(s) repeated along x, the last axis of every field's grid."""
    a = a.reshape(-1, nx)
    return np.ascontiguousarray(np.concatenate([a, a], axis=1))


@pytest.mark.parametrize("codec", sorted(EPS))
@pytest.mark.parametrize("shape", SHAPES)
def test_odd_rows_equal_repeated_even_rows(oracle_mod, shape, codec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    nx, ny, nz = shape
    o, f, g, S = start(oracle_mod, shape)
    a = sim.Simulation(shape, lattice="D3Q19", precision=codec, diag_every=2, **PRM)
    b = sim.Simulation((2 * nx, ny, nz), lattice="D3Q19", precision=codec, diag_every=2, **PRM)
    a.set_state(f, g, S, 0)
    b.set_state(twice(f, nx), twice(g, nx), twice(S, nx), 0)
    f, g, S = a.get_state()
    o.set_state(f, g, S, 0)
    a.step(1)
    o.step(1)
    fa, ga, Sa = a.get_state()
    fo, go, So = o.get_state()
    eps, fmov = EPS[codec], np.abs(fo[1:]).max()
    # a few roundings of the offsets plus FP32 arithmetic
    assert np.abs(fa - fo).max() <= 4 * eps * fmov + 1e-6 * np.abs(fo).max()
    assert np.abs(ga - go).max() <= 8 * eps * np.abs(go).max()
    a.step(3)
    b.step(4)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(twice(x, nx).ravel(), y.ravel())
    ma, mb = a.moments(), b.moments()
    for k in ma:
        assert np.array_equal(twice(ma[k], nx).ravel(), mb[k].ravel())
    da, db = a.last_diagnostics(), b.last_diagnostics()
    assert da["u_max"] == db["u_max"] and da["mu_min"] == db["mu_min"]
    assert np.isclose(2 * da["sum_phi"], db["sum_phi"], rtol=1e-12)
    a.close()
    b.close()
