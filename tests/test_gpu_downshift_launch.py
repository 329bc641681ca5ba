"""The downshifted step's launches: particle counts at the edges of a tile and
of several tiles per CTA (particles are independent, so a run of the first n
equals the larger run's first n bit for bit, history included), and a DoF that
is not finite (its tets' particles freeze with status NONFINITE where they
stand, as under the plain step; the others are untouched)."""
import numpy as np
import pytest

from paper_2208_12795_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64, MIXED, Q24 = 0, 1, 2
MOST = 152 * 3 * 256 + 300


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_12795_gb300 import build
    build.build()


def _run(prec, n, steps=3, bad_edge=None, offset=0):
    from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState
    wl = I.te101_cavity(5, MOST, 200.0, 1e4, 1, 21, dt=2e-9, ramp_sigma=0.0, jitter=0.2)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    st = ParticleState.from_host(wl.particles.subset(n), prec)
    for k in ("x", "vx", "tet"):
        t = getattr(st, k)
        setattr(st, k, torch.empty(n + offset, dtype=t.dtype, device="cuda")[offset:].copy_(t))
    env.locate(st)
    tet0 = st.tet.cpu().numpy()
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    if bad_edge is not None:
        e[bad_edge] = complex(float("inf"), 0.0)
    ds = Downshift(env, n)
    for k in range(steps):
        ds.step(st, e, b, 1.0, wl.omega0, k * wl.dt, wl.dt)
        env.deposit(wl.omega0, (k + 1) * wl.dt)
    g = st.to_numpy()
    g["planes"] = ds.planes[:33].cpu().numpy()
    g["tet0"], g["x0"], g["te"] = tet0, wl.particles.x[:n], env.query()["tet_edges"]
    return g


@pytest.fixture(scope="module")
def largest():
    return {prec: _run(prec, MOST) for prec in (FP64, MIXED, Q24)}


@pytest.mark.parametrize("n,offset", [(1, 0), (255, 0), (257, 1), (1030, 0)])
@pytest.mark.parametrize("prec", [FP64, MIXED, Q24])
def test_first_particles_of_a_larger_run(largest, prec, n, offset):
    g, big = _run(prec, n, offset=offset), largest[prec]
    assert big["n_cross"].sum() > MOST // 4
    for k in ("x", "y", "z", "vx", "vy", "vz", "tet", "status", "n_cross"):
        assert np.array_equal(g[k], big[k][:n]), k
    assert np.array_equal(g["planes"], big["planes"][:, :n])


@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_dof_not_finite_freezes_its_tets(prec):
    good = _run(prec, 3000, steps=1)
    bad = _run(prec, 3000, steps=1, bad_edge=200)
    hit = (good["te"][good["tet0"]] == 200).any(1)
    assert 0 < hit.sum() < 1500
    assert (bad["status"][hit] == 3).all() and np.array_equal(bad["tet"][hit], -2 - good["tet0"][hit])
    assert np.array_equal(bad["x"][hit], good["x0"][hit])
    for k in ("x", "vx", "tet", "status"):
        assert np.array_equal(bad[k][~hit], good[k][~hit]), k


def test_first_step_captured_leaves_nothing_to_the_replay():
    """A first step that is only captured (its graph never replayed) and the
    same steps launched after it: the run of a new integrator."""
    from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState
    n = 2000
    wl = I.te101_cavity(5, MOST, 200.0, 1e4, 1, 21, dt=2e-9, ramp_sigma=0.0, jitter=0.2)
    env = FempicEnv.from_mesh(wl.mesh, precision=MIXED)
    st = ParticleState.from_host(wl.particles.subset(n), MIXED)
    env.locate(st)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    env.push_step(st, e, b, 0.0, wl.omega0, 0.0, wl.dt, out=st.empty_like())   # the env's own scratch
    env.deposit(wl.omega0, wl.dt)
    ds = Downshift(env, n)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        ds.step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt)
    ds.started = False
    for k in range(3):
        ds.step(st, e, b, 1.0, wl.omega0, k * wl.dt, wl.dt)
    want, got = _run(MIXED, n), st.to_numpy()
    for k in got:
        assert np.array_equal(got[k], want[k]), k
