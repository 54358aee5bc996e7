"""Longer prefix pieces, at most as many as CTAs: where the nodes are alike; not
where short nodes hold the CTAs and a long node's piece would be the tail."""
import pytest

from paper_2608_24658_gb300 import _lib
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests.test_plan import verify_plan


def _tree(mode, d, h_q, prefix, nodes, node_len, branches, tokens):
    """branches under each of `nodes` nodes (under the prefix itself if 0)"""
    parent, lens, leaves = [-1], [prefix], []
    forks = []
    for _ in range(nodes):
        forks.append(len(parent))
        parent.append(0)
        lens.append(node_len)
    for f in forks or [0]:
        for _ in range(branches):
            leaves.append(len(parent))
            parent.append(f)
            lens.append(tokens)
    return W.build_tree("pieces", parent, lens, leaves, num_q_heads=h_q, num_kv_heads=8,
                        head_dim=d, mode=mode, values=False)


def _wide_pages(tree):
    with Plan.for_tree(tree, host_only=True, num_sms=152) as plan:
        verify_plan(tree, plan)
        items = plan.export(_lib.TABLE_ITEMS)[plan.export(_lib.TABLE_WIDE_QUEUE)]
        return items[:, 1], plan.info()


@pytest.mark.parametrize("h_q", [32, 64])
def test_short_nodes_do_not_lengthen_the_prefix(h_q):
    """256 pages of prefix in one piece were 75.6 (81.2) us of a step that takes
    42.5 (53.5) with pieces of a CTA's share."""
    pages, _ = _wide_pages(_tree("bf16", 128, h_q, 4096, 8, 64, 16, 300))
    assert pages.max() <= 128


@pytest.mark.parametrize("mode,d,h_q,prefix,nodes,node_len,branches,tokens,entries", [
    ("bf16", 64, 64, 16384, 4, 100, 16, 350, 128),     # 32 tiles of 1024 pages in 3, and 32 of 7
    ("fp8", 128, 32, 16384, 8, 1024, 8, 150, 144),     # 16 of 1024 in 5, and 64 of 64
])
def test_alike_nodes_are_lengthened(mode, d, h_q, prefix, nodes, node_len, branches, tokens, entries):
    pages, info = _wide_pages(_tree(mode, d, h_q, prefix, nodes, node_len, branches, tokens))
    assert len(pages) == entries
    assert info["num_wide_ctas"] == entries
