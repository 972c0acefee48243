"""Kernels launched beside the end of their predecessor (programmatic dependent
launches), read from the sources: a race between launches cannot be provoked
on purpose."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_02917_gb300", "csrc")
WAIT = re.compile(r"\b(?:umma::grid_dependency_wait|cs_chain)\(\)")


def functions(text):
    """(name, parameter list, body) of every function definition."""
    text = re.sub(r"__(?:launch_bounds|maxnreg)__\([^()]*\)", "", text)
    for m in re.finditer(r"^[^\n#/]*\b(\w+)\(([^;{}]*)\)[^;{}]*\{\s*$", text, re.M):
        depth, i = 1, m.end()
        while depth and i < len(text):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), m.group(2), re.sub(r"//[^\n]*", "", text[m.end():i])


DEPENDENT = {}
for _path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
    if not _path.endswith("umma.cuh"):
        for _name, _params, _body in functions(open(_path).read()):
            if WAIT.search(_body) and _name != "cs_chain":
                DEPENDENT[_name] = (_params, _body)


def test_the_kernels_are_found():
    assert set(DEPENDENT) == {"llt_kernel", "lltt_body", "gemv_t_lat_kernel", "gemv_n_lat_kernel", "lanczos_kernel",
                              "npga_step_body", "adj_proj_kernel", "adj_finish_kernel", "cs_count_kernel",
                              "cs_scan_kernel", "cs_fill_kernel", "cs_sort_kernel", "cs_tn_kernel",
                              "gemm_chunk_kernel"}


# A block of the sketch's tail with no quarter to form may leave: the launch ends with the blocks that wait.
@pytest.mark.parametrize("name", sorted(set(DEPENDENT) - {"gemm_chunk_kernel"}))
def test_no_way_out_before_the_wait(name):
    body = DEPENDENT[name][1]
    first = WAIT.search(body).start()
    assert not re.search(r"\breturn\b(?! Elem)", re.sub(r"\[&\][^{};]*\{[^{}]*\}", "", body[:first]))


# Inputs of the calls and vectors complete before the predecessor started (the Lanczos q_j: two products back).
# Everything else a dependent kernel reads may be written while it is already alive, so the read-only path
# (const __restrict__, __ldg) is closed to it; __ldcg is a coherent load that stays behind the wait.
SETTLED = {"L", "Lt", "h", "sign", "rs", "row_scale", "cscale", "qj"}


@pytest.mark.parametrize("name", sorted(DEPENDENT))
def test_no_read_only_loads_of_a_running_predecessors_output(name):
    params, body = DEPENDENT[name]
    for p in re.findall(r"\bconst\s+[\w:]+\s*\*\s*__restrict__\s*(\w+)", params):
        if p in SETTLED:
            continue
        uses = re.findall(rf"(?<!\.)\b{p}\b", body)
        assert len(uses) == len(re.findall(rf"__ldcg\({p}\b", body)), f"{name}: {p}"
    for expr in re.findall(r"__ldg\((\w+)", body):
        assert expr in SETTLED, f"{name}: __ldg({expr}"
