"""CPU check of the sources: kernels that are launched chained (launch.cuh)
start before their predecessors end, so that read-only loads (__ldg, const
__restrict__ parameters), which the language allows only for data that is
constant over a kernel's lifetime, are kept for what no chained kernel writes:
the mode table and the plan (its axes, sorted cells and permutation)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2212_10961_gb300", "csrc")
# bases of a pointer into the mode table or the plan
CONSTANT = re.compile(r"^(&?p\.(hot|cold)|p\.[XYZ]|d\.[XYZ]|gg\.[XYZ]|[XYZ]|cold|cells(\[c\])?|src\[[^\]]+\]|a\.p|perm|d\.perm|"
                      r"args\.(cold|hot|order|kpref)|o\.table_kpref|axes|xs|ys|zs)(?!\w)")
PARAMETERS = {"cold", "hot", "xs", "ys", "zs", "perm"}


def _functions(text):
    """(name, head, body) of every function definition at namespace level."""
    text = re.sub(r"__launch_bounds__\((?:[^()]|\((?:[^()]|\(\))*\))*\)\s*", "", text)
    for m in re.finditer(r"\n((?:template <[^>]*>\n)?(?:__global__|__device__)[^;{]*?(\w+)\(([^{;]*)\))\s*\{\n", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(2), m.group(1), text[m.end():i]


def _sources():
    return {f: open(os.path.join(CSRC, f)).read() for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh"))}


def _chained():
    names = set()
    for text in _sources().values():
        for call in re.findall(r"launch_chained\(([^;]*?);", text):
            names |= set(re.findall(r"\b(\w+_kernel|grid_split_finalize|synth_split_finalize)\b", call))
    return names


def test_the_chained_kernels_are_found():
    assert {"band_select_kernel", "band_line_kernel", "grid_adj_kernel", "loss_sum_kernel", "synth_split_finalize",
            "band_cells_kernel", "bwd_reduce_kernel"} <= _chained()


@pytest.mark.parametrize("name", sorted(_sources()))
def test_read_only_loads_of_chained_kernels(name):
    chained, found = _chained(), 0
    for fn, head, body in _functions(_sources()[name]):
        if "__global__" in head:
            if fn not in chained:
                continue
            assert "pdl_wait();" in body or "grid_mma_body<" in body, fn
            for p in re.findall(r"const \w+\s*\*\s*__restrict__ (\w+)", head):
                assert p in PARAMETERS, "%s: %s" % (fn, p)
        elif name in ("synth_fwd.cu", "synth_bwd.cu", "plan.cu", "maps.cu"):
            continue  # helpers of kernels that are launched in full
        for arg in re.findall(r"__ldg\(((?:reinterpret_cast<[^>]*>\()?[^;]*)", body):
            found += 1
            assert CONSTANT.match(arg), "%s: __ldg(%s" % (fn, arg[:60])
    if name == "band.cu":
        assert found >= 8
