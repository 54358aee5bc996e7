"""The tcgen05 prefix tile at head_dim 64: tiles of 17 to 129 rows, nodes that
end in every part of a 64-token block, pages in pool order and permuted, NaN
past every node's end."""
import numpy as np
import pytest

import oracle
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests import parity as PT

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("h_q,h_kv,branches", [(1, 1, 17), (4, 1, 5), (8, 2, 32), (8, 1, 16), (3, 1, 43)])
def test_prefix_tile_d64(h_q, h_kv, branches, permute):
    # requests whose prefixes end around the edges of a block and of a piece
    prefixes = [1, 16, 63, 64, 65, 130, 700]
    parent, lens, leaves = [], [], []
    for n in prefixes:
        root = len(parent)
        parent.append(-1)
        lens.append(n)
        for b in range(branches):
            parent.append(root)
            lens.append(1 + (7 * b) % 40)
            leaves.append(len(parent) - 1)
    tree = W.build_tree("prefix_d64", parent, lens, leaves, num_q_heads=h_q, num_kv_heads=h_kv,
                        head_dim=64, seed=8, permute_pages=permute, extra_pages=3,
                        tail_value=float("nan"), device="cuda")
    PT.nan_fill_unused_pages(tree)
    with Plan.for_tree(tree) as plan:
        assert plan.info()["num_wide_items"] > 0
        out, lse = plan.decode_tree(tree)
        plan.check()
    ref_o, ref_l = oracle.decode(**oracle.tree_kwargs(tree.to("cpu")))
    PT.compare(tree, out, lse, ref_o, ref_l, None, tree.name)
