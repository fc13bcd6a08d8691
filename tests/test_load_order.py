"""How the kernels with overlapped launches read what another kernel writes: never through the non-coherent path, and
by nothing that the compiler may move across the wait for the kernel before."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_05423_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_no_non_coherent_loads_of_data():
    for name in ("pp_arith.cuh", "pp_lines.cuh", "pp_hlines.cuh", "pp_hx.cuh", "pp_zpart.cu", "pp_zsing.cuh"):
        assert "ld.global.nc" not in _code(name), name
    for name in ("pp_arith.cuh", "pp_lines.cuh"):
        assert "__ldg" not in _code(name), name
    # tables that the plan wrote before any launch: twiddles, mode descriptors, multipliers
    tables = {"pp_hlines.cuh": {"reinterpret_cast<const int4*>(p)", "reinterpret_cast<const float2*>(p)"},
              "pp_zpart.cu": {"reinterpret_cast<const int4*>(m)", "reinterpret_cast<const float4*>(m) + 1",
                              "a.qtab + m->qoff + k0 + i"},
              "pp_zsing.cuh": {"wt + r", "wt + i"}}
    for name, allowed in tables.items():
        code = _code(name)
        found = re.findall(r"__ldg\(((?:[^()]|\((?:[^()]|\([^()]*\))*\))*)\)", code)
        assert found and set(found) <= allowed, (name, found)
    hl = _code("pp_hlines.cuh")  # the two casts above are those of the twiddle types
    assert set(re.findall(r"hld\(const (\w+)\* p\)", hl)) == {"htwa", "htwb"}


def test_loads_stay_behind_the_wait():
    for name in sorted(os.listdir(CSRC)):
        for volatile, body in re.findall(r"\basm\s*(volatile)?\s*\(((?:[^()]|\((?:[^()]|\([^()]*\))*\))*)\)\s*;", _code(name)):
            if "ld.global" in body or "griddepcontrol" in body:
                assert volatile and '"memory"' in body, (name, body)
