"""The downshifted step over several tiles per CTA: while one tile's particles
are worked on, the next one's state and history are copied into the same shared
buffer.  Particles are independent, so those around every wave of CTAs and the
last, ragged tile equal a run of their own (one tile per CTA) bit for bit,
history included: with the 16-byte copies (n a multiple of 4, aligned arrays),
with an odd n, and with arrays off the 16-byte boundary."""
import numpy as np
import pytest

from paper_2208_12795_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64, MIXED, Q24 = 0, 1, 2
WAVE = 152 * 3 * 256          # particles of one wave of CTAs of the mixed kernel
N = 3 * WAVE + 300            # three tiles per CTA and a ragged fourth in some


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_12795_gb300 import build
    build.build()


@pytest.fixture(scope="module")
def load():
    return I.te101_cavity(5, N + 1, 200.0, 1e4, 1, 22, dt=2e-9, ramp_sigma=0.0, jitter=0.2)


def _run(wl, prec, lo, hi, offset=0):
    from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState
    P, n = wl.particles, hi - lo
    part = I.Particles(*(getattr(P, k)[lo:hi] for k in ("x", "y", "z", "vx", "vy", "vz")),
                       np.array([0, n], np.int64), P.q, P.m, P.w)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    st = ParticleState.from_host(part, prec)
    for k in ("x", "vx", "tet"):
        t = getattr(st, k)
        setattr(st, k, torch.empty(n + offset, dtype=t.dtype, device="cuda")[offset:].copy_(t))
    env.locate(st)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    ds = Downshift(env, n)
    for k in range(4):
        ds.step(st, e, b, 1.0, wl.omega0, k * wl.dt, wl.dt)
        env.deposit(wl.omega0, (k + 1) * wl.dt)
    return st.to_numpy(), ds.planes[:33].cpu().numpy()


@pytest.mark.parametrize("n,offset", [(N, 0), (N + 1, 0), (N, 1)])
@pytest.mark.parametrize("prec", [FP64, MIXED, Q24])
def test_later_tiles_equal_their_own_run(load, prec, n, offset):
    big, planes = _run(load, prec, 0, n, offset)
    assert big["n_cross"].sum() > n // 4
    for lo in (WAVE - 500, 2 * WAVE - 500, 3 * WAVE - 800, n - 1000):
        own, own_planes = _run(load, prec, lo, lo + 1000)
        for k, v in own.items():
            assert np.array_equal(v, big[k][lo:lo + 1000]), (k, lo)
        assert np.array_equal(own_planes, planes[:, lo:lo + 1000]), lo
