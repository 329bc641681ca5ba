"""A run that injects particles: the crossing queue holds whole tiles of 256, so
a step on a set grown inside its last tile needs no new scratch, and one that
has been outgrown is made an eighth larger.  Such steps can be captured into a
graph (which neither synchronizes nor allocates) and equal the steps launched."""
import numpy as np
import pytest

from paper_2208_12795_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64, MIXED, Q24 = 0, 1, 2


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_12795_gb300 import build
    build.build()


@pytest.mark.parametrize("prec", [FP64, MIXED, Q24])
@pytest.mark.parametrize("eager,captured", [
    ((1,), 2), ((255,), 256), ((5000,), 5001), ((4865,), 5120),   # inside the last tile
    ((5000, 5121), 5761),          # outgrown: ceil(5121 * 9/8 / 256) * 256 = 5888
    ((77, 300, 5121), 5888),
])
def test_a_grown_set_steps_without_new_scratch(prec, eager, captured):
    from paper_2208_12795_gb300.env import FempicEnv, ParticleState
    wl = I.workload_hot_small(n_particles=6000)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()

    def load(n):
        st = ParticleState.from_host(wl.particles.subset(n), prec)
        env.locate(st)
        return st

    for n in eager:
        env.push_step(load(n), e, b, 1.0, wl.omega0, 0.0, wl.dt)
    want, got = load(captured), load(captured)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        env.push_step(got, e, b, 1.0, wl.omega0, 0.0, wl.dt)
    graph.replay()
    env.push_step(want, e, b, 1.0, wl.omega0, 0.0, wl.dt)
    w, g = want.to_numpy(), got.to_numpy()
    for k in w:
        assert np.array_equal(w[k], g[k]), k
