"""A block may write a peer's shared memory only once the peer runs: every
device function that exchanges over a cluster passes a cluster barrier first
(read from the sources; the hazard cannot be provoked on purpose)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_02917_gb300", "csrc")
# what writes into peers: the projector's exchanges, the adjoint's sums, the fused pass's and the pair kernels' pushes
EXCHANGE = re.compile(r"\bP\.(?:prepare|solve|reduce_\w+)\(|\bcluster_sums<|\bst_async_v\d\(|\bmbar_arrive_cluster\(|\btma_load_2d_pair\(")
BARRIER = re.compile(r"\bcluster_wait<CL>\(\)|\bcluster_barrier<CL>\(\)|\bcluster\.sync\(\)|this_cluster\(\)\.sync\(\)")


def functions(text):
    """(name, body) of every function definition whose body starts a line-ending brace."""
    for m in re.finditer(r"^[^\n#/]*\b(\w+)\([^;{}]*\)[^;{}]*\{\s*$", text, re.M):
        depth, i = 1, m.end()
        while depth and i < len(text):
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), re.sub(r"//[^\n]*", "", text[m.end():i])


def exchanging():
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"__(?:launch_bounds|maxnreg)__\([^()]*\)", "", open(path).read())
        for name, body in functions(text):
            if re.search(r"ClusterProj<CL> P\{|cluster_sums<CL, \d+>\(|st_async_v\d\(llt|tma_load_2d_pair\(", body):
                out.append((os.path.basename(path), name, body))
    return out


FOUND = exchanging()


def test_the_kernels_are_found():
    names = {n for _, n, _ in FOUND}
    assert {"npga_step_body", "npga_bt_step_body", "init_x_body", "frontier_init_kernel", "frontier_step_kernel",
            "project_batch_kernel", "adj_proj_kernel", "llt_kernel", "lltt_body", "gemm_chunk_pair_kernel",
            "sigma_pair_kernel"} <= names


@pytest.mark.parametrize("which", [f"{f}:{n}" for f, n, _ in FOUND])
def test_cluster_barrier_before_the_first_exchange(which):
    body = {f"{f}:{n}": b for f, n, b in FOUND}[which]
    first = EXCHANGE.search(body).start()
    barrier = BARRIER.search(body)
    assert barrier is not None and barrier.start() < first
    if "cluster_wait<CL>()" in barrier.group():
        assert "cluster_arrive<CL>()" in body[:barrier.start()]
