"""The FP64 tile march of the D2Q9 step against the oracle at the sizes where
its columns and rows can go wrong: the last strip one or two columns wide (its
stencil then reaches columns past the grid), strips just short of 128 columns,
odd and single rows (an iteration holds two), grids narrower than the stencil.

Tolerance: 1e-12 of a field's largest magnitude plus 1e-14 of the state's, the
FP64 bound of the parity tests (about 100 roundings of the O(1) populations).
"""
import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=4.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=20.0, rho_v=1.0, nu_l=0.6, nu_v=0.1,
           Gx=1e-6, Gy=-2e-6)


@pytest.mark.parametrize("shape", [(126, 5), (127, 9), (128, 2), (129, 7), (130, 3), (131, 1),
                                   (2, 2), (1, 1), (33, 30), (257, 31)])
def test_fp64_march_against_oracle(oracle_mod, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    nx, ny = shape
    o = oracle_mod.Oracle(shape, **PRM)
    o.init_phi(wl.droplet(nx, ny, 0.3 * min(nx, ny) + 1.0, 4.0))
    f, g, S = o.get_state()
    g = g + wl.perturbed_state(g.shape, 1e-3, 11)
    S = S + wl.perturbed_state(S.shape, 1e-4, 12)
    o.set_state(f, g, S, 0)
    s = sim.Simulation(shape, precision="fp64", diag_every=3, **PRM)
    s.set_state(f, g, S, 0)
    s.step(7)
    o.step(6)
    d6 = o.diag()
    o.step(1)
    got, ref = s.get_state(), o.get_state()
    atol = 1e-14 * max(np.abs(ref[0]).max(), np.abs(ref[1]).max())
    mg, mo = s.moments(), o.macros()
    for a, b in list(zip(got, ref)) + [(mg[k], mo[k]) for k in ("phi", "mu", "p", "u")]:
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max() + atol
    d = s.last_diagnostics()  # of the state at step 6
    N = nx * ny
    assert d["step"] == 6 and not d["nonfinite"]
    assert abs(d["sum_phi"] - d6["sum_phi"]) <= 1e-12 * abs(d6["sum_phi"]) + N * atol
    assert abs(d["u_max"] - d6["umax"]) <= 1e-12 * d6["umax"] + 4 * atol
    s.close()


@pytest.mark.parametrize("shape", [(16, 128), (17, 33), (31, 2), (1, 1), (3, 5), (48, 50), (150, 29),
                                   (2431, 1)])
def test_small_grid_kernel_equals_march(oracle_mod, shape):
    """Grids of at most 152 tiles of 16 x 2 nodes take a kernel that splits the
    node update over four warps.  Its expressions are those of the tile march,
    which the same flow takes when it is repeated in y (periodic) until it has
    more tiles: the same bits, and the oracle's step within the FP64 bound."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    nx, ny = shape
    tiles = lambda h: ((nx + 15) // 16) * ((h + 1) // 2)  # noqa: E731
    times = 1
    while tiles(ny * times) <= 152:
        times += 1
    assert tiles(ny) <= 152
    o = oracle_mod.Oracle(shape, **PRM)
    o.init_phi(wl.droplet(nx, ny, 0.3 * min(nx, ny) + 1.0, 4.0))
    f, g, S = o.get_state()
    g = g + wl.perturbed_state(g.shape, 1e-3, 13)
    S = S + wl.perturbed_state(S.shape, 1e-4, 14)
    o.set_state(f, g, S, 0)
    rep = lambda a: np.concatenate([a.reshape(-1, ny, nx)] * times, axis=1)  # noqa: E731
    a = sim.Simulation(shape, precision="fp64", **PRM)
    b = sim.Simulation((nx, ny * times), precision="fp64", **PRM)
    a.set_state(f, g, S, 0)
    b.set_state(rep(f), rep(g), rep(S), 0)
    a.step(5)
    b.step(5)
    o.step(5)
    got, ref = a.get_state(), o.get_state()
    atol = 1e-14 * max(np.abs(ref[0]).max(), np.abs(ref[1]).max())
    for x, y, z in zip(got, b.get_state(), ref):
        assert np.array_equal(rep(x).ravel(), y.ravel())
        assert np.abs(x - z).max() <= 1e-12 * np.abs(z).max() + atol
    a.close()
    b.close()
