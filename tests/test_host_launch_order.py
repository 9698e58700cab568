"""What a kernel that is launched before the work ahead of it has ended may touch of the caller's, read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_12990_b200", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def test_batch_projections_know_the_experts_from_the_plan_alone():
    """The gate/up launch of a batch is resident while the routing, or whatever else is ahead, still runs.  The caller's expert
    tables are read by the plan kernel, behind its wait; the projections get no pointer to them."""
    text = _source("batch.cu")
    params = text[text.index("struct BParams {"):]
    assert "slicemoe_expert" not in params[:params.index("};")]
    body = text[text.index("batch_ffn_kernel(const __grid_constant__"):]
    before = body[:body.index("b_dep_wait();")]
    assert "p.ctl" not in before and "p.segs" not in before and "p.head" not in before
    plan = text[text.index("batch_plan_kernel(const BPlanParams"):]
    before = plan[:plan.index("b_dep_wait();")]
    assert re.findall(r"\bp\.\w+", before) == []


def test_weights_are_complete_before_a_layer_kernel_starts():
    """The decode kernel streams the shared experts' slices ahead of its wait.  So a kernel that writes slices lets nobody start
    while it runs: neither pack nor those that expand a slice for the second tier."""
    for name in ("pack.cu", "tier.cu"):
        assert "launch_dependents" not in _source(name), name
