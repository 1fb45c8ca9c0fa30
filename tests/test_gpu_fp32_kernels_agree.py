"""A single FP32 D2Q9 run mixes kernels: plain steps of grids up to 640 000 nodes take
the one-tile kernel, steps with fused diagnostics the march, batches the march
with one launch per step or many.  One step from one state gives the same bits
through each, at tile edges and on a grid of many tiles.
"""
import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=4.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=20.0, rho_v=1.0, nu_l=0.6, nu_v=0.1,
           Gx=1e-6, Gy=-2e-6)


@pytest.mark.parametrize("shape", [(64, 4), (65, 5), (3, 7), (301, 203), (1000, 640)])
def test_one_step_gives_the_same_bits_through_every_kernel(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, sim
    build.build()
    nx, ny = shape
    plain = sim.Simulation(shape, precision="fp32", **PRM)
    plain.init_phi(wl.two_droplets(nx, ny, 0.2 * min(nx, ny) + 1.0, 4.0))
    plain.step(20)
    f, g, S = plain.get_state()
    g = g + wl.perturbed_state(g.shape, 1e-3, 31)
    S = S + wl.perturbed_state(S.shape, 1e-4, 32)

    def stepped(s, step):
        s.set_state(f, g, S, 0)
        step(1)
        return s.get_state()

    want = stepped(plain, plain.step)
    assert all(np.isfinite(w).all() for w in want)
    diag = sim.Simulation(shape, precision="fp32", diag_every=1, **PRM)
    got = {"diagnostics step": stepped(diag, diag.step)}
    batch = sim.Batch([(shape, PRM)], precision="fp32")
    for width in (64, 128):
        batch.set_shape(width, 16)
        got[f"batch step, width {width}"] = stepped(batch.case(0), batch.step)
    for k, v in got.items():
        for a, b in zip(want, v):
            assert np.array_equal(a, b), k
    # several steps: per-step launches against multi-step launches
    plain.set_state(f, g, S, 0)
    plain.step(6)
    want = plain.get_state()
    batch.set_shape(64, 16)
    batch.set_persistent(True)
    batch.case(0).set_state(f, g, S, 0)
    batch.step(6)
    batch.sync()
    for a, b in zip(want, batch.case(0).get_state()):
        assert np.array_equal(a, b)
    for x in (plain, diag, batch):
        x.close()
