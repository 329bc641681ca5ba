"""A downshift handle made for one precision form holds that form's per-tet
tables alone; a step on an env of the other kind makes its own."""
import ctypes as C

import numpy as np
import pytest

from paper_2208_12795_gb300 import build, capi, inputs as I

FP64, MIXED, Q24 = 0, 1, 2


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def test_bad_arguments_rejected_on_host():
    lib = capi.load()
    h = C.c_void_p()
    assert lib.fempic_downshift_create_form(None, 0, C.byref(h)) == capi.FEMPIC_EINVAL
    nodes = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], float)
    tets = np.array([[0, 1, 2, 3]], np.int32)
    d = capi.fempic_mesh_desc(4, 1, nodes.ctypes.data, tets.ctypes.data, (C.c_double * 3)(0, 0, 0),
                              (C.c_double * 3)(1, 1, 1))
    for form in (-1, 3):
        assert lib.fempic_downshift_create_form(C.byref(d), form, C.byref(h)) == capi.FEMPIC_EINVAL
        assert "form" in capi.fempic_downshift_last_error() and not h.value


# Bytes per tet: geometry, edge and face ids 136; then tables and coefficients
# 32 f64 (FP64) or 32 f64 + 24 f32 (mixed).  Five allocations, each rounded up
# to 2 MiB.
@pytest.mark.gpu
@pytest.mark.parametrize("prec,per_tet", [(FP64, 136 + 256), (MIXED, 136 + 352), (Q24, 136 + 352)])
def test_memory_of_one_form(prec, per_tet):
    torch = pytest.importorskip("torch")
    from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState
    wl = I.te101_cavity(24, 64, 200.0, 1e4, 1, 21, dt=2e-9, ramp_sigma=0.0)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    st = ParticleState.from_host(wl.particles, prec)
    env.locate(st)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    first = Downshift(env, st.n)          # the process's and the env's own scratch
    first.step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    ds = Downshift(env, st.n)
    ds.step(st, e, b, 1.0, wl.omega0, wl.dt, wl.dt)
    torch.cuda.synchronize()
    used = free0 - torch.cuda.mem_get_info()[0]
    assert used <= per_tet * env.n_tets + 5 * (2 << 20), used / env.n_tets


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [FP64, MIXED, Q24])
@pytest.mark.parametrize("made_for", [None, FP64, MIXED, Q24])
def test_any_handle_steps_any_form(prec, made_for):
    torch = pytest.importorskip("torch")
    from paper_2208_12795_gb300.env import Downshift, FempicEnv, ParticleState, _mesh_desc
    wl = I.workload_hot_small(n_particles=600)
    got = []
    for handle in (None, made_for):
        env = FempicEnv.from_mesh(wl.mesh, precision=prec)
        st = ParticleState.from_host(wl.particles, prec)
        env.locate(st)
        e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
        b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
        ds = Downshift(env, st.n)
        if got:
            ds.close()
            desc = _mesh_desc(*env._mesh)
            ds.h = (capi.fempic_downshift_create(desc) if handle is None
                    else capi.fempic_downshift_create_form(desc, handle))
        for k in range(4):
            ds.step(st, e, b, 1.0, wl.omega0, k * wl.dt, wl.dt)
        got.append((st.to_numpy(), ds.planes[:33].cpu().numpy()))
    (a, pa), (c, pc) = got
    for k in a:
        assert np.array_equal(a[k], c[k]), k
    assert np.array_equal(pa, pc)
