"""The steps of a batch read what the steps before them wrote from any thread block, so each step ends at a
point where all blocks meet: a kernel's end where every step is a launch, a cluster-wide barrier in the
kernel of small batches, a grid-wide one in a group's persistent kernel.  A missing one shows only under an
unlucky schedule, so the order is checked in the source (no GPU needed)."""
import os
import re

import pytest

from paper_1811_09136_gb300 import _build

STEPS = ["k_classify", "k_plan", "k_commit", "k_rehash_big", "k_rehash_huge", "k_insert", "k_units", "k_order"]


def kernels_source():
    with open(os.path.join(_build.CSRC, "rept_kernels.cuh")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def function_body(source, name):
    """The text between the braces of the function `name`."""
    at = source.index("{", re.search(r"\b%s\(" % name, source).end())
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(source[end], 0)
        if depth == 0:
            return source[at:end]
        end += 1


@pytest.mark.parametrize("kernel,barrier", [("k_state", "cluster_barrier"), ("k_group_persistent", "grid_barrier")])
def test_all_blocks_meet_between_the_steps_of_one_launch(kernel, barrier):
    body = function_body(kernels_source(), kernel)
    calls = re.findall(r"\b(k_\w+)_body\(|\b(%s)\(" % barrier, body)
    order = [step or met for step, met in calls]
    assert [x for x in order if x != barrier] == STEPS
    for step, following in zip(STEPS, STEPS[1:]):
        between = order[order.index(step) + 1:order.index(following)]
        assert between == [barrier], f"{kernel}: {step} and {following} are separated by {between}"


def test_cluster_barrier_takes_warps_that_have_not_met():
    """The steps end in divergent code; the .aligned barrier is undefined for such a warp."""
    body = function_body(kernels_source(), "cluster_barrier")
    assert "barrier.cluster.arrive.release;" in body and "barrier.cluster.wait.acquire;" in body


def test_memory_that_a_launch_writes_is_not_read_through_the_read_only_path():
    """The intersection may be resident while the inserts write the pool, and the persistent kernel writes the
    pool and the prefixes itself: neither may be read with loads for data that stays unwritten throughout."""
    source = kernels_source()
    assert not re.search(r"__ldg\b|\.global\.nc", source)
    for name in ("table_slot", "table_find", "group_prefix_body", "intersect_group_body", "group_stream_search",
                 "k_group_persistent"):
        params = re.search(r"\b%s\((.*?)\)\s*\{" % name, source, re.S).group(1)
        for param in params.split(","):
            if re.search(r"\b(table|pref|cursor|pc)$", param):
                assert "__restrict__" not in param, f"{name}: {param.strip()}"
