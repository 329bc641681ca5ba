"""fempic_debug_stall stays in force over steps that have no staged push kernel
(into another set, downshifted) and is used up by the next step of a mixed form
in place, with one level or three."""
import pytest

from paper_2208_12795_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [1, 3])
@pytest.mark.parametrize("prec", [1, 2])
def test_stall_waits_for_its_kernel(prec, levels):
    from paper_2208_12795_gb300 import build, capi
    build.build()
    from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState
    wl = I.workload_hot_small(n_particles=600)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    st = ParticleState.from_host(wl.particles, prec)
    env.locate(st)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    ds = Downshift(env, st.n)
    capi.fempic_debug_stall(env.h, 0, 1_000_000)
    env.push_step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt, out=st.empty_like())
    ds.step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt)
    assert env.error_count()[0]

    def step():
        if levels == 1:
            env.push_step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt)
        else:
            env.push_step3(st, [e] * 3, [b] * 3, (1.0, 0.0, 0.0), 1.0, wl.omega0, 0.0, wl.dt)

    step()
    assert not env.error_count()[0]
    step()
    assert env.error_count()[0]
