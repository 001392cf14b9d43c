"""Bulk copies read and write memory through the async proxy, which a
__threadfence or a barrier does not order against ordinary stores.  In the
persistent batched kernels the adjoint phase bulk-copies the packed traces that
other CTAs of the same launch stored, into shared memory that the forward items
wrote; a missing fence is a race that a run need not show, so the source is
checked for it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2404_10928_gb300", "csrc")


def function_body(name):
    """The text of the function `name` of pa_ops.cu, braces matched, without comments."""
    with open(os.path.join(CSRC, "pa_ops.cu"), encoding="utf-8") as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    m = re.search(r"\b" + name + r"\([^;{]*\)\s*\{", text)
    assert m, name
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return m.group(0), text[m.end():i - 1]


def test_grid_barrier_fences_both_sides():
    head, body = function_body("grid_barrier")
    assert "bool to_bulk" in head
    fence = r"if \(to_bulk\) fence_proxy_async\(\);"
    assert re.search(r"^\s*" + fence + r"\s*__syncthreads\(\);", body)
    assert re.search(r"__syncthreads\(\);\s*" + fence + r"\s*$", body)
    assert "fence.proxy.async" in function_body("fence_proxy_async")[1]


@pytest.mark.parametrize("kernel", ["k_batch_landweber", "k_batch_cgls"])
def test_adjoint_phases_follow_a_fenced_barrier(kernel):
    _, body = function_body(kernel)
    # barriers and adjoint items in the order of the text, which is their order in
    # the launch (loop bodies end in a barrier)
    events = re.findall(r"grid_barrier\(([^;]*)\);|(adj_landweber_block|adj_norm_block)<", body)
    assert sum(bool(adj) for _, adj in events) >= 1
    for before, (_, adj) in zip(events, events[1:]):
        if adj:
            assert before[0] and before[0].split(",")[-1].strip() == "true", before


def test_barriers_are_invalidated_before_their_memory_is_used_again():
    """A batched CTA calls adj_accumulate once per item: its mbarriers' memory is
    initialised again, and holds the forward's windows in between, which PTX allows
    only after mbarrier.inval."""
    _, body = function_body("adj_accumulate")
    m = re.search(r"if \(!PLAIN && tid == 0\) \{(.*?)\n  \}\s*__syncthreads\(\);\s*return", body, re.S)
    assert m
    assert {"mbar_inval(&s_full[i]);", "mbar_inval(&s_empty[i]);"} <= set(
        re.findall(r"mbar_inval\([^)]*\);", m.group(1)))
    assert "mbar_wait" not in m.group(1) and "mbar_wait" not in body[m.end():]
