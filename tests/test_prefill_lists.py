"""e4m3 prefill plans on both sides of the rule that gives a pair its whole path
as one list of pages: every query row sees its ancestors and its own tokens once."""
import pytest

from paper_2608_24658_gb300 import _lib
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests.test_prefill_plan import CASES, verify_prefill_plan


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("sms", [1, 2, 152])
def test_e4m3_lists_cover(name, sms):
    t = CASES[name]()
    t8 = W.build_prefill(name, t.parent, t.node_len, t.leaf_node, num_q_heads=t.num_q_heads,
                         num_kv_heads=t.num_kv_heads, head_dim=128, mode="fp8", values=False)
    with Plan.for_prefill(t8, host_only=True, num_sms=sms) as plan:
        verify_prefill_plan(t8, plan)


@pytest.mark.parametrize("chunks,lists", [(4, True), (5, False)])
def test_e4m3_list_rule(chunks, lists):
    """4 pairs on one SM read whole paths, 5 a run per node."""
    t = W.build_prefill("rule", [-1] + [0] * chunks, [50] + [20] * chunks,
                        list(range(1, chunks + 1)), num_q_heads=4, num_kv_heads=1, head_dim=128,
                        mode="fp8", values=False)
    with Plan.for_prefill(t, host_only=True, num_sms=1) as plan:
        verify_prefill_plan(t, plan)
        rng = plan.export(_lib.TABLE_MERGE_RANGES)
        assert ((rng[:, 1] - rng[:, 0] == 1).all()) == lists


@pytest.mark.parametrize("sms,lists", [(31, False), (32, True), (152, True)])
def test_e4m3_many_pairs_read_whole_paths(sms, lists):
    """More than 4 pairs an SM: whole paths but on a small partition."""
    n = 5 * 152 // 4
    t = W.build_prefill("many", [-1, 0] + [1] * n, [70, 9] + [1 + k % 3 for k in range(n)],
                        list(range(2, 2 + n)), num_q_heads=4, num_kv_heads=4, head_dim=128,
                        mode="fp8", values=False)
    with Plan.for_prefill(t, host_only=True, num_sms=sms) as plan:
        verify_prefill_plan(t, plan)
        assert plan.info()["num_wide_items"] // 2 >= 5 * sms
        rows = plan.export(_lib.TABLE_STREAM_ROWS)
        assert (rows & 15).any() == lists          # a node's end inside an item
