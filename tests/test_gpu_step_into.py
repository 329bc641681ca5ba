"""fempic_push_step_to takes two sets of one species table that share no memory:
any array of the one on any of the other (the same one, another one, a view
shifted by some elements) and differing charges, masses or weights are EINVAL
before any launch; sets that lie side by side in one allocation are accepted."""
import copy

import numpy as np
import pytest

from paper_2208_12795_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP64, MIXED = 0, 1
N = 600


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2208_12795_gb300 import build
    build.build()


def _setup(prec):
    from paper_2208_12795_gb300.env import FempicEnv, ParticleState
    wl = I.workload_hot_small(n_particles=N)
    env = FempicEnv.from_mesh(wl.mesh, precision=prec)
    st = ParticleState.from_host(wl.particles, prec)
    env.locate(st)
    e = torch.from_numpy(wl.e_tilde).to(env.dof_dtype).cuda()
    b = torch.from_numpy(wl.b_tilde).to(env.dof_dtype).cuda()
    return wl, env, st, lambda dst: env.push_step(st, e, b, 1.0, wl.omega0, 0.0, wl.dt, out=dst)


def _refused(env, st, dst, step, match):
    from paper_2208_12795_gb300 import capi
    before = st.to_numpy()
    steps = env.stats()["steps"]
    with pytest.raises(capi.FempicError, match=match):
        step(dst)
    assert env.stats()["steps"] == steps
    for k, v in st.to_numpy().items():
        assert np.array_equal(v, before[k]), k


@pytest.mark.parametrize("prec", [FP64, MIXED])
@pytest.mark.parametrize("name", ["x", "y", "z", "vx", "vy", "vz", "tet", "status", "n_cross"])
def test_a_shared_array_is_refused(prec, name):
    _, env, st, step = _setup(prec)
    dst = st.empty_like()
    setattr(dst, name, getattr(st, name))
    _refused(env, st, dst, step, "overlap")


@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_shifted_and_crossed_views_are_refused(prec):
    _, env, st, step = _setup(prec)
    for name in ("x", "vz", "tet", "status"):
        t = getattr(st, name)
        for shift in (1, N - 1):
            both = torch.empty(N + shift, dtype=t.dtype, device="cuda")
            setattr(st, name, both[:N].copy_(t))
            for lo, hi in ((0, shift), (shift, 0)):   # in before out, and behind it
                setattr(st, name, both[lo:lo + N].copy_(t.clone()))
                dst = st.empty_like()
                setattr(dst, name, both[hi:hi + N])
                _refused(env, st, dst, step, "overlap")
    dst = st.empty_like()
    dst.y = st.z                                      # another array of the set
    _refused(env, st, dst, step, "overlap")


@pytest.mark.parametrize("prec", [FP64, MIXED])
@pytest.mark.parametrize("name", ["q", "m", "w"])
def test_another_species_table_is_refused(prec, name):
    _, env, st, step = _setup(prec)
    dst = copy.copy(st.empty_like())
    setattr(dst, name, getattr(st, name) * 2.0)
    _refused(env, st, dst, step, "species tables differ")


@pytest.mark.parametrize("prec", [FP64, MIXED])
def test_sets_side_by_side_in_one_allocation(prec):
    _, env, st, step = _setup(prec)
    want, dst = st.empty_like(), st.empty_like()
    step(want)
    for name in ("x", "y", "z", "vx", "vy", "vz", "tet", "status", "n_cross"):
        t = getattr(st, name)
        both = torch.empty(2 * N, dtype=t.dtype, device="cuda")
        setattr(st, name, both[:N].copy_(t))
        setattr(dst, name, both[N:])
    step(dst)
    w, g = want.to_numpy(), dst.to_numpy()
    for k in w:
        assert np.array_equal(w[k], g[k]), k
