"""Orders in the kernels' sources that no run can show to be missing (a race may never show): another
CTA's shared memory is touched only behind a meeting of the cluster, an operator call reads the maps and
the samples only behind its dependency wait, and tensor memory is held before a successor may start."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1411_6206_gb300", "csrc")


def code(name):
    """A source without its comments."""
    with open(os.path.join(CSRC, name)) as f:
        s = f.read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def body(src, name):
    """Body of the function `name` defined in src."""
    m = re.search(re.escape(name) + r"\([^;{}]*\)\s*\{", src)
    assert m, f"{name} is not defined"
    depth = 0
    for i in range(m.end() - 1, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[m.end():i]
    raise AssertionError(f"{name} does not end")


@pytest.mark.parametrize("file,function", [("k_eig.cu", "gram_share"), ("k_dc_reg.cu", "k_dc_reg"),
                                           ("k_dc_fixed.cu", "k_dc_fixed"), ("k_dc_rows.cuh", "dc_rows_plane")])
def test_cluster_meets_before_remote_shared_memory(file, function):
    b = body(code(file), function)
    first = b.index("map_shared_rank")
    assert re.search(r"cl\.sync\(\)|cluster_wait\(\)", b[:first]), "remote access before the cluster has met"


def test_eigen_kernel_pairs_its_cluster_barrier():
    """Every CTA arrives before it waits for its predecessors, and no path leaves between the arrive and
    the wait."""
    b = body(code("k_eig.cu"), "k_eig")
    assert b.index("cluster_arrive()") < b.index("pdl_wait()")
    before = b[b.index("cluster_arrive()"):b.index("gram_share<CL>(a, sh, nn, n, 0")]
    for m in re.finditer(r"\breturn;", before):
        near = before[max(0, m.start() - 60):m.start()]
        assert "cluster_wait()" in near or "gram_share<CL>" in near, near


@pytest.mark.parametrize("file,function,first_read", [("k_dc_reg.cu", "k_dc_reg", "load_col(grp)"),
                                                      ("k_dc_fixed.cu", "k_dc_fixed", "issue(grp, "),
                                                      ("k_dc_rows.cuh", "dc_rows_plane", "stage_samples(rank)")])
def test_operator_calls_wait_before_they_read_maps_or_samples(file, function, first_read):
    """Outside a frame (no control block) the call may directly follow the kernel that wrote them."""
    b = body(code(file), function)
    assert "if (!a.ctrl) pdl_wait();" in b[:b.index(first_read)]


@pytest.mark.parametrize("function", ["k_gram_tc", "k_reproj_tc"])
def test_tensor_memory_is_held_before_the_successor_is_released(function):
    """A later launch must not take the tensor memory that a CTA of this one still waits for: the warp that
    allocates is the one that releases, afterwards."""
    src = code("k_tc.cu")
    b = body(src, function)
    assert "pdl_trigger()" not in b and "tmem_alloc(" not in b
    assert "if (warp == 0) alloc_and_release(tslot);" in b[:b.index("pdl_wait()")]
    r = body(src, "alloc_and_release")
    assert r.index("tmem_alloc(") < r.index("pdl_trigger()")
