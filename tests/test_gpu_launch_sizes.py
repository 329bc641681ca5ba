"""Particle counts at the edges of the common path's launches (one particle,
one warp, a tile less or more one, several tiles per CTA with a ragged last
one) and particle arrays off the 16-byte boundary bulk copies need, against
the FP64 oracle.

Zero field and dt = 2^-31 s, so that both sides track and deposit the same
straight segments: tets, crossing counts, positions and velocities bit-exact,
G within 1e-12 of its maximum (the deposit's bound of the identical-endpoint
tests)."""
import numpy as np
import pytest

from oracle.oracle import OracleMesh, OracleState, push_step as oracle_push
from paper_2208_12795_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64, MIXED = 0, 1
DT = 2.0 ** -31
SIZES = (1, 32, 255, 256, 257, 1000, 152 * 4 * 256 + 77)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_12795_gb300 import build
    build.build()


@pytest.fixture(scope="module")
def oracle_run():
    mesh = I.kuhn_cube_mesh(6, jitter=0.2, rng=np.random.default_rng(31))
    n = max(SIZES)
    rng = np.random.default_rng(8)
    pos = rng.uniform(0.0, 1.0, size=(n, 3))
    v = (rng.standard_normal((n, 3)) * 1e8).astype(np.float32).astype(np.float64)
    parts = I.Particles(pos[:, 0], pos[:, 1], pos[:, 2], v[:, 0], v[:, 1], v[:, 2],
                        np.array([0, n], np.int64), np.array([-I.E_CHARGE]), np.array([I.M_ELECTRON]),
                        np.array([1e3]))
    om = OracleMesh(mesh.nodes, mesh.tets, mesh.lo, mesh.hi)
    tet0, _ = om.locate(parts.x, parts.y, parts.z)
    out = {}
    for k in SIZES:
        sub = parts.subset(k)
        ost = OracleState(sub, tet0[:k])
        G = np.zeros(om.n_edges)
        z = np.zeros(om.n_edges, np.complex128), np.zeros(om.n_faces, np.complex128)
        for s in range(2):
            oracle_push(om, ost, *z, 0.0, 1.3e9, s * DT, DT, G)
        out[k] = sub, ost, G
    return mesh, out


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_counts_and_alignment(oracle_run, prec, offset, n):
    from paper_2208_12795_gb300.env import FempicEnv, ParticleState
    mesh, runs = oracle_run
    parts, ost, oG = runs[n]
    env = FempicEnv.from_mesh(mesh, precision=prec)
    st = ParticleState.from_host(parts, prec)
    for k in ("x", "y", "z", "vx", "vy", "vz", "tet"):   # the same values, one element past an aligned start
        t = getattr(st, k)
        w = torch.empty(n + offset, dtype=t.dtype, device="cuda")[offset:]
        setattr(st, k, w.copy_(t))
    env.locate(st)
    e = torch.zeros(env.n_edges, dtype=env.dof_dtype, device="cuda")
    b = torch.zeros(env.n_faces, dtype=env.dof_dtype, device="cuda")
    G = torch.zeros(env.n_edges, dtype=torch.float64, device="cuda")
    for s in range(2):
        env.push_step(st, e, b, 0.0, 1.3e9, s * DT, DT)
        env.deposit(1.3e9, (s + 1) * DT, G_cum_out=G)
    g = st.to_numpy()
    for k in ("tet", "n_cross", "status", "x", "y", "z"):
        assert np.array_equal(g[k], getattr(ost, k)), k
    for k in ("vx", "vy", "vz"):
        assert np.array_equal(g[k].astype(np.float64), getattr(ost, k)), k
    assert np.abs(G.cpu().numpy() - oG).max() <= 1e-12 * np.abs(oG).max()
    assert env.error_count()[0]


@pytest.mark.parametrize("n", [1, 257, 5000])
@pytest.mark.parametrize("prec", [FP64, MIXED, 2])
def test_step_into_another_set_equals_the_step_in_place(prec, n):
    """Walls that absorb, a crossing cap, a NaN velocity, an out-of-range and a
    missing tet: every array of the other set comes out as the step in place
    leaves it, and the set stepped from is unchanged."""
    from paper_2208_12795_gb300 import capi
    from paper_2208_12795_gb300.env import FempicEnv, ParticleState
    wl = I.workload_hot_small(n_particles=5000, wall_mode=1)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec, wall_mode=1, max_crossings=2)
    st = ParticleState.from_host(wl.particles.subset(n), prec)
    env.locate(st)
    if n > 100:
        st.vy[7] = float("nan")
        st.tet[11] = env.n_tets + 3
        st.tet[12] = -1
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    env.push_step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt)   # some particles are frozen already
    src, dst = st.to_numpy(), st.empty_like()
    env.push_step(st, e, b, 1.0, wl.omega0, wl.dt, wl.dt, out=dst)
    for k, v in st.to_numpy().items():
        assert np.array_equal(v, src[k], equal_nan=True), k
    env.push_step(st, e, b, 1.0, wl.omega0, wl.dt, wl.dt)
    got = dst.to_numpy()
    assert n < 100 or (got["status"] != 0).sum() > 100
    for k, v in st.to_numpy().items():
        assert np.array_equal(v, got[k], equal_nan=True), k
    with pytest.raises(capi.FempicError, match="overlap"):
        env.push_step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt, out=st)


@pytest.mark.parametrize("prec", [FP64, MIXED, 2])
def test_captured_steps_replay(prec):
    """Two steps with their deposits captured in a CUDA graph (the launches
    overlap their set-up) and replayed: the state and G_cum of the same steps
    launched one by one."""
    from paper_2208_12795_gb300.env import FempicEnv, ParticleState
    wl = I.workload_hot_small(n_particles=3000)
    got = []
    for captured in (False, True):
        env = FempicEnv.from_mesh(wl.mesh, precision=prec)
        st = ParticleState.from_host(wl.particles, prec)
        env.locate(st)
        e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
        b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
        G = torch.zeros(env.n_edges, dtype=torch.float64, device="cuda")

        def steps():
            for k in range(2):
                env.push_step(st, e, b, 1.0, wl.omega0, k * wl.dt, wl.dt)
                env.deposit(wl.omega0, (k + 1) * wl.dt, G_cum_out=G)

        steps()   # the first calls allocate
        torch.cuda.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                steps()
            for _ in range(3):
                graph.replay()
        else:
            for _ in range(3):
                steps()
        got.append((st.to_numpy(), G.cpu().numpy()))
    (a, Ga), (c, Gc) = got
    for k in a:
        assert np.array_equal(a[k], c[k]), k
    assert np.abs(Ga - Gc).max() <= 1e-13 * np.abs(Ga).max()


@pytest.mark.parametrize("prec", [FP64, MIXED, 2])
def test_fewer_particles_never_allocate(prec):
    """After a step on a set, steps on smaller ones (whose launches take other
    tiles and more regions) can be captured: their scratch is the larger set's."""
    from paper_2208_12795_gb300.env import FempicEnv, ParticleState
    sizes = (152 * 2 * 256 - 256, 152 * 2 * 128 - 1, 5000, 33)
    wl = I.workload_hot_small(n_particles=sizes[0] + 1)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()

    def load(n):
        st = ParticleState.from_host(wl.particles.subset(n), prec)
        env.locate(st)
        return st

    env.push_step(load(sizes[0] + 1), e, b, 1.0, wl.omega0, 0.0, wl.dt)
    for n in sizes:
        want, got = load(n), load(n)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            env.push_step(got, e, b, 1.0, wl.omega0, 0.0, wl.dt)
        graph.replay()
        env.push_step(want, e, b, 1.0, wl.omega0, 0.0, wl.dt)
        w, g = want.to_numpy(), got.to_numpy()
        for k in w:
            assert np.array_equal(w[k], g[k]), (n, k)
