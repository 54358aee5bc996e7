"""The e4m3 prefix tile's order of work: prefix CTAs that run several items each,
with items of one block up to more blocks than are left when the next item is
pulled (8), in queue order of mixed lengths, NaN past every node's end."""
import pytest

import oracle
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prefixes", [[1, 64], [63, 511, 512], [65, 513, 577, 1100], [16]])
@pytest.mark.parametrize("h_q,h_kv,branches", [(16, 2, 5), (2, 2, 18)])
def test_many_prefix_items_per_cta(h_q, h_kv, branches, prefixes):
    parent, lens, leaves = [], [], []
    for n in prefixes * (48 // len(prefixes)):
        root = len(parent)
        parent.append(-1)
        lens.append(n)
        for b in range(branches):
            parent.append(root)
            lens.append(6000 // branches + (37 * b) % 90)
            leaves.append(len(parent) - 1)
    tree = W.build_tree("prefix_e4m3", parent, lens, leaves, num_q_heads=h_q, num_kv_heads=h_kv,
                        head_dim=128, mode="fp8", seed=9, extra_pages=3,
                        tail_value=float("nan"), device="cuda")
    PT.nan_fill_unused_pages(tree)
    with Plan.for_tree(tree) as plan:
        info = plan.info()
        assert info["num_wide_items"] >= 2 * info["num_wide_ctas"]
        out, lse = plan.decode_tree(tree)
        plan.check()
    ref_o, ref_l = oracle.decode(**oracle.tree_kwargs(tree.to("cpu")))
    PT.compare(tree, out, lse, ref_o, ref_l, None, tree.name)
