"""CPU test of the loads in kernels that are launched dependently (programmatic dependent launch).

Such a kernel is resident while the launch before it still runs, and that launch may write the
state, the references and the porosity it reads behind its wait.  The read-only load (__ldg, or a
load through a `const * __restrict__` kernel parameter, which the compiler may turn into one) is for
data that no one writes during the whole life of the kernel, and nothing keeps it behind the wait.
Whether a compiled kernel goes wrong on it is chance, so the rule is checked in the source."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_5929_gb300", "csrc")

# parameters that only the host writes, by a copy in stream order: block lists, instance constants
HOST_WRITTEN = {"inst", "blocks"}


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _dependent_kernels(text):
    """(name, parameters, body) of every kernel that waits for the launch before it."""
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(([^{;]*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        body = text[m.end():i]
        if "griddepcontrol.wait" in body or "pdl_enter()" in body or "tile_steps(" in body:
            yield m.group(1), m.group(2), body


@pytest.mark.parametrize("name,kernels", [
    ("lbm_f32.cu", {"k_two", "k_step", "k_fields", "k_batch_step", "k_tile"}),
    ("lbm_16.cu", {"k_step16", "k_fields16", "k_batch_step16"}),
    ("fno_net.cu", {"k_pack", "k_pack_many", "k_fwd", "k_proj", "k_bwd", "k_r2k", "k_k2r", "k_mixf", "k_mixb"}),
])
def test_no_read_only_parameters(name, kernels):
    found = {}
    for kernel, params, body in _dependent_kernels(_source(name)):
        found[kernel] = [p for p in re.findall(r"const[^,()]*\*\s*__restrict__\s+(\w+)", params) if p not in HOST_WRITTEN]
        assert "__ldg(" not in body
    assert set(found) == kernels
    assert not any(found.values()), found


@pytest.mark.parametrize("name", ["lbm_two.cuh", "lbm_step32.cuh", "lbm_tile.cuh", "lbm_f32.cu", "lbm_16.cu",
                                  "fno_net.cu", "tc.cuh"])
def test_no_read_only_loads(name):
    assert "__ldg(" not in _source(name) and "ld.global.nc" not in _source(name)


def test_shared_node_updates_load_by_kind_of_launch():
    """lbm_nodes.cuh also serves kernels of ordinary launches: its loads take the kind of launch, and
    the dependent kernels ask for theirs."""
    nodes, dep = _source("lbm_nodes.cuh"), _source("lbm_16.cu")
    assert nodes.count("__ldg(") == 1 and re.search(r"if constexpr \(DEP\) return \*p;\s*else return __ldg\(p\);", nodes)
    assert not re.search(r"\b(ldv|ld2|ldq2)\s*\(", dep)
    assert not re.search(r"wall_state<STO, float>|update_pair<STO, VEC>", dep)
    assert len(re.findall(r"wall_state<STO, float, LAY_N, true>", dep)) == 2
