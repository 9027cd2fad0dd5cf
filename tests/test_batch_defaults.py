"""BatchPlan.configure() with no arguments asks for what a new plan has."""
import inspect
import os
import re

import paper_1905_03277_gb300 as hm


def test_configure_defaults_are_the_plans():
    src = open(os.path.join(os.path.dirname(hm.__file__), "csrc", "batch.cu")).read()
    plan = src[src.index("struct hmfsr_batch_plan_t {"):src.index("cudaGraphExec_t exec")]

    def field(name):
        return eval(re.search(r"\b%s = ([^,;]+)[,;]" % name, plan).group(1))

    got = {k: v.default for k, v in inspect.signature(hm.BatchPlan.configure).parameters.items() if k != "self"}
    want = dict(merge_tile_w="mw", ctas_per_sm="ctas_per_sm", regs_variant="regs_variant", queue_order="order",
                spin_limit="spin_limit", inject_stall="inject_stall")
    assert got == {k: field(v) for k, v in want.items()}
