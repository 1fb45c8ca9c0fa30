"""The offset formats' scales after a diagnostics refresh: the power of two from
the largest stored offset, wherever it lies (the scan reads eight values at a
time: first and last elements, remainders of 1 to 7 values, fields smaller than
one block's share)."""
import math

import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=5.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=10.0, rho_v=1.0, nu_l=1.0, nu_v=0.1)


def pad(b):
    return (b + 255) // 256 * 256


def parts(buf, N):
    """(h bits, k bits, scales) of a checkpoint's payload."""
    fb, gb = pad(19 * N * 2) + pad(7 * N * 4) + 256, 19 * N * 2
    raw = buf.view(np.uint8)[len(buf) - (fb + gb + 4 * N):]
    sc = raw[fb - 256:fb - 248].copy().view(np.float32)
    return (raw[:19 * N * 2].copy().view(np.uint16), raw[fb:fb + gb].copy().view(np.uint16), sc)


@pytest.mark.parametrize("shape", [(5, 3, 1), (8, 8, 4), (33, 9, 5), (64, 40, 20)])
@pytest.mark.parametrize("where", ["first", "last", "middle"])
@pytest.mark.parametrize("codec", ["f16off", "bf16off"])
def test_refreshed_scales(shape, where, codec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, capi, sim
    build.build()
    nx, ny, nz = shape
    N = nx * ny * nz
    s = sim.Simulation(shape, lattice="D3Q19", precision=codec, **PRM)
    s.init_phi(wl.two_droplets(nx, ny, min(shape) / 4 + 1.0, 5.0, nz=nz))
    s.step(2)
    # a large offset at one place of h (population 1 is +x, 18 is (0, -y, -z)) and of k
    for field, value in ((0, 0.4), (1, 0.2)):
        i, (x, y, z) = {"first": (0, (0, 0, 0)), "last": (18, (nx - 1, -2, -2)),
                        "middle": (9, (nx // 2, ny // 2, nz // 2))}[where]
        n = ((z % nz) * ny + y % ny) * nx + x % nx
        assert capi.lbm_debug_poke(s.handle, field, i, n, value) == capi.LBM_OK
    h, k, sc = parts(s.save(), N)
    dec = (lambda u: np.array([u], np.uint16).view(np.float16).astype(np.float32)[0]) \
        if codec == "f16off" else \
        (lambda u: (np.array([u], np.uint32) << 16).view(np.float32)[0])
    want = []
    for v, c in ((h, sc[0]), (k, sc[1])):
        m = float(dec((v & 0x7fff).max())) * float(c)
        want.append(max(2.0 ** -16, math.ldexp(1.0, math.frexp(m / 4096.0)[1])) if m > 0 else 2.0 ** -16)
    if where == "last":  # the poke is the field's last element
        assert (h[-1] & 0x7fff) == (h & 0x7fff).max()
    s.diagnostics()
    s.step(1)
    got = parts(s.save(), N)[2]
    assert [float(v) for v in got] == want
    s.close()
