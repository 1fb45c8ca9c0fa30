"""The initial condition of the offset storage (D3Q19), beside the runs that
start from it."""
import numpy as np
import pytest

from paper_2311_10827_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PRM = dict(W=5.0, M=0.05, alpha=1.0, sigma=1e-3, rho_l=10.0, rho_v=1.0, nu_l=1.0, nu_v=0.1)


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10827_gb300 import build, capi, sim
    build.build()
    return torch, capi, sim


def on_caller_buffers(env, shape, precision):
    """A context on state buffers that the test holds."""
    torch, capi, sim = env
    params = sim.make_params(precision, **PRM)
    rc, (fb, gb, sb) = capi.lbm_state_bytes(shape, capi.LBM_D3Q19, params)
    assert rc == capi.LBM_OK
    bufs = [torch.zeros(n, dtype=torch.uint8, device="cuda") for n in (fb, fb, gb, gb, sb)]
    torch.cuda.synchronize()
    rc, h = capi.lbm_create_with_buffers(shape, capi.LBM_D3Q19, params, bufs)
    assert rc == capi.LBM_OK
    return sim.Simulation(shape, lattice="D3Q19", precision=precision, _borrow=h, **PRM), bufs


@pytest.mark.parametrize("buffer", [1, 3])
@pytest.mark.parametrize("precision", ["f16off", "bf16off", "fp32", "fp64"])
@pytest.mark.parametrize("shape", [(40, 24, 20), (33, 9, 5)])
def test_phi_may_lie_in_the_other_state_buffers(env, shape, precision, buffer):
    """lbm_init_phi initialises buffers 0; a caller that owns the state memory can
    hand over phi in f or g buffer 1, which are free until the first step."""
    torch, capi, sim = env
    phi0 = wl.droplet(shape[0], shape[1], 6.0, PRM["W"], nz=shape[2])
    a, bufs = on_caller_buffers(env, shape, precision)
    b = sim.Simulation(shape, lattice="D3Q19", precision=precision, **PRM)
    N = int(np.prod(shape))
    phi = bufs[buffer][:8 * N].view(torch.float64)
    phi.copy_(torch.tensor(phi0.ravel(), device="cuda"))
    torch.cuda.synchronize()
    a.init_phi(phi)
    b.init_phi(phi0)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    a.step(3)
    b.step(3)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    capi.lbm_destroy(a.handle)
    b.close()


C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
for _a, _b in ((0, 1), (0, 2), (1, 2)):
    for _s in ((1, 1), (1, -1), (-1, 1), (-1, -1)):
        _v = [0, 0, 0]
        _v[_a], _v[_b] = _s
        C3.append(tuple(_v))


@pytest.mark.parametrize("size", [1e-39, 1e-3])
@pytest.mark.parametrize("precision", ["f16off", "bf16off"])
def test_initial_offsets_round_once(env, precision, size):
    """The stored moving offsets of an initial field are (f - f^eq)/s rounded to FP32
    and then to 16 bits, also where f - f^eq is below the smallest normal FP32
    value (the scale s = 2^-16 lifts it back into the range of BF16)."""
    torch, capi, sim = env
    shape, N = (20, 6, 5), 600
    rng = np.random.default_rng(5)
    phi0 = size * rng.uniform(0.5, 1.5, shape[::-1])
    s, bufs = on_caller_buffers(env, shape, precision)
    s.init_phi(phi0)
    s.sync()
    raw = bufs[0].cpu()
    h = raw[:38 * N].view(torch.int16).numpy().reshape((19,) + phi0.shape)
    off = (38 * N + 255) // 256 * 256
    mu_f = raw[off:off + 8 * N].view(torch.float32).numpy()[N:].reshape(phi0.shape)
    at = lambda a, c: np.roll(a, (-c[2], -c[1], -c[0]), axis=(0, 1, 2))  # noqa: E731
    d = [at(phi0, c) - phi0 for c in C3]
    lap = sum(d[1:7]) / 3.0 + sum(d[7:]) / 6.0
    mu = 4.0 * s.beta * (phi0 - 1.0) * phi0 * (phi0 - 0.5) - s.kappa * lap
    for i, c in enumerate(C3):
        if i == 0:
            continue
        w = 1.0 / 18.0 if i < 7 else 1.0 / 36.0
        eq = (np.float32(w) * (np.float32(s.alpha) * mu_f)).astype(np.float64)
        v = torch.tensor(((at(w * s.alpha * mu, c) - eq) * 65536.0).astype(np.float32))
        want = v.to(torch.float16 if precision == "f16off" else torch.bfloat16).view(torch.int16)
        assert np.array_equal(h[i], want.numpy())
    capi.lbm_destroy(s.handle)
