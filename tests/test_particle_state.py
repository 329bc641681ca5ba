"""The particle set's C structure names the species arrays it holds, also
after they are replaced and in copies (their addresses are taken when the
arrays are set)."""
import copy
import pickle

import numpy as np
import pytest

torch = pytest.importorskip("torch")


def _state():
    from paper_2208_12795_gb300.env import ParticleState
    cols = [torch.zeros(4, dtype=torch.float64) for _ in range(6)]
    return ParticleState(*cols, [0, 1, 4], [1.0, 2.0], [3.0, 4.0], [5.0, 6.0])


@pytest.mark.parametrize("how", [lambda s: s, copy.copy, copy.deepcopy, lambda s: pickle.loads(pickle.dumps(s)),
                                 lambda s: s.empty_like()], ids=["itself", "copy", "deepcopy", "pickle", "empty_like"])
def test_cstruct_addresses(how):
    st = how(_state())
    for replaced in (False, True):
        if replaced:
            st.q, st.species_begin = np.array([7.0, 8.0]), np.array([0, 2, 4], np.int64)
        c = st.cstruct()
        assert (c.n, c.n_species, c.x, c.vz, c.tet) == (4, 2, st.x.data_ptr(), st.vz.data_ptr(), st.tet.data_ptr())
        assert (c.status, c.n_cross) == (st.status.data_ptr(), st.n_cross.data_ptr())
        for k in ("species_begin", "q", "m", "w"):
            assert getattr(c, k) == getattr(st, k).ctypes.data, k
