"""Kernels launched with programmatic stream serialization are resident while
the kernels before them still write, so the non-coherent load path (__ldg, or a
const __restrict__ parameter), which promises memory that does not change while
the kernel runs, is for the tables that are fixed once per mesh.  Read from the
CUDA sources: every such load names one of those tables."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_12795_gb300", "csrc")
FILES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))

# tables built when an env or a downshift handle is made: geometry, its
# products, FP32 gradients, node, edge and face ids, neighbours, adjacency
FIXED = {"geom", "geom64", "tgeo", "dgeo", "grad32", "tetrec", "tn", "nb", "te", "tf", "estart", "eslot", "fslot"}
# local names of pointers into them, by the function that forms them
LOCAL = {"ld_geo": {"rec"}, "ld_glo": {"rec"}, "ldg_int4": {"p"}, "ld_tet_geo": {"a", "b"},
         "k_ds_push_mixed": {"x0"}, "cross64_advance": {"g"}, "k_ds_field32": {"D", "g1"}}


def _source(name):
    txt = open(os.path.join(CSRC, name)).read()
    txt = re.sub(r"/\*.*?\*/", " ", txt, flags=re.S)
    return re.sub(r"//[^\n]*", "", txt)


def _functions(txt):
    """(name, parameters, body) of every function defined at namespace level."""
    for m in re.finditer(r"^[^\n#;]*?\b(\w+)\(((?:[^()]|\([^()]*\))*)\)\s*\{", txt, flags=re.M):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(txt[i], 0)
            i += 1
        yield m.group(1), m.group(2), txt[m.end():i]


def _launched():
    names = set()
    for f in FILES:
        names |= set(re.findall(r"\blaunch\((k_\w+)", _source(f)))
        names |= set(re.findall(r"[?:]\s*\(?(?:\w+ \? )?(k_\w+)<", _source(f)))
    return names


def test_the_step_kernels_are_found():
    names = _launched()
    assert {"k_field_f32", "k_push_mixed", "k_ds_push_mixed", "k_cross_df", "k_dof_grad", "k_tet_finalize"} <= names


@pytest.mark.parametrize("name", FILES)
def test_parameters(name):
    launched = _launched()
    for fn, params, _ in _functions(_source(name)):
        if fn not in launched:
            continue
        for par in re.findall(r"const \w+\* __restrict__ (\w+)", params):
            assert par in FIXED, (fn, par)


@pytest.mark.parametrize("name", FILES)
def test_loads(name):
    for fn, _, body in _functions(_source(name)):
        if fn == "k_ds_permute":   # an ordinary launch
            continue
        for arg in re.findall(r"__ldg\(&?((?:\w+\.)?\w+)", body):
            base = arg.split(".")[-1]
            assert base in FIXED or base in LOCAL.get(fn, ()), (fn, arg)


def test_local_names_point_into_fixed_tables():
    """What LOCAL lists: callers pass, or the function forms, a fixed table's address."""
    env, ds = _source("fempic_env.cu"), _source("fempic_downshift.cu")
    for call in re.findall(r"\b(?:ld_geo|ld_glo)\((\w+(?:\.\w+)?),", env):
        assert call in ("A.tetrec", "geo"), call          # geo: bary_q_at, called with A.tetrec
    for call in re.findall(r"\bbary_q_at\((\S+),", env):
        assert call in ("A.tetrec",), call
    for call in re.findall(r"\bldg_int4\(&A\.(\w+)", env):
        assert call in ("nb", "tn"), call
    for txt in (env, ds):
        for geom, tgeo in re.findall(r"\bld_tet_geo\((\w+), (\w+),", txt):
            assert geom in FIXED and tgeo in FIXED, (geom, tgeo)
    bodies = {fn: body for txt in (env, ds) for fn, _, body in _functions(txt)}
    assert "x0 = reinterpret_cast<const double*>(A.tetrec" in bodies["k_ds_push_mixed"]
    assert "g = A.geom64" in bodies["cross64_advance"]
    assert "D = reinterpret_cast<const double2*>(dgeo" in bodies["k_ds_field32"] and "g1 = geom" in bodies["k_ds_field32"]
