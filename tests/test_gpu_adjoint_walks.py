"""Walks of the deposited-current adjoint at the edges of its list: one
particle, a warp's worth, more than a warp's, more than a CTA's, on steps of
about 0.8 of the cube, so that nearly every particle walks many tets and
reflects several times (the Jacobian of the reflections before the last one).
FP64 form against the oracle's tangent.

Bound: the tangent of one step perturbs by about 1e-4 of the gradient for an
FP32 ulp of the path on steps a quarter as long (near-grazing crossings), which
is 2e-13 for an FP64 ulp; four times the crossings and reflections may multiply
it by some tens per step, so 1e-10 of sum |g_i d_i| leaves room for rounding
alone."""
import numpy as np
import pytest

from oracle.oracle import OracleMesh
from paper_2208_12795_gb300 import inputs as I
from test_gpu_current_adjoint import FP64, _directions, _gpu, _mag, _mods, _oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 32, 33, 300])
def test_long_walks_match_oracle_tangent(n):
    A, _, _ = _mods()
    wl = I.te101_cavity(4, 300, 300.0, 1e3, 4, 12, dt=80e-9, ramp_sigma=0.0, jitter=0.2)
    P = wl.particles.subset(n)
    rng = np.random.default_rng(5)
    u = rng.standard_normal(OracleMesh(wl.mesh.nodes, wl.mesh.tets).n_edges)
    env, st0, e, b, sch, L, eg, bg, adj = _gpu(wl, P, FP64, 2, 2, u)
    tet0 = st0.tet.cpu().numpy()
    for _ in range(3):
        de, db, tr, tv = _directions(rng, wl, P.n, env.n_edges, env.n_faces)
        Lo, jv, status, scale = _oracle(wl, P, tet0, 2, u, de, db, tr, tv, 0, 4096)
        assert abs(L - Lo) <= 1e-12 * scale
        assert abs(A.grad_dot(eg, bg, adj, de, db, tr, tv) - jv) <= 1e-10 * _mag(eg, bg, adj, de, db, tr, tv)
