"""The suffix piece length: whatever the nodes' lengths, the pieces cover them and
are never more than 2.5 pieces per warp make (more partial rows than that would
not fit the scratch such plans had)."""
import numpy as np
import pytest

from paper_2608_24658_gb300 import _lib
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests.test_plan import verify_plan

WARPS = {("fp8", 128): 12, ("bf16", 128): 8, ("bf16", 64): 8}


def _tree(mode, d, lens, h_kv):
    return W.build_tree("suffix_lengths", [-1] + [0] * len(lens), [2048] + list(lens),
                        list(range(1, len(lens) + 1)), num_q_heads=8 * h_kv, num_kv_heads=h_kv,
                        head_dim=d, mode=mode, seed=2, values=False)


@pytest.mark.parametrize("mode,d", sorted(WARPS))
@pytest.mark.parametrize("lens", [[3000] * 40, list(range(100, 4000, 61)), [16] * 64, [1] * 17,
                                  [60000] * 24, [40, 9000]])
@pytest.mark.parametrize("sms", [1, 152])
def test_pieces_bounded(mode, d, lens, sms):
    tree = _tree(mode, d, lens, 8)
    with Plan.for_tree(tree, host_only=True, num_sms=sms) as plan:
        verify_plan(tree, plan)
        items = plan.export(_lib.TABLE_ITEMS)[plan.export(_lib.TABLE_NARROW_QUEUE)]
    if 8 * len(lens) <= 16:                   # the prefix is suffix work too
        lens = [2048] + lens
    pages = 8 * np.array([-(-n // 16) for n in lens])
    shortest = max(4, min(128, int(pages.sum() / (2.5 * sms * WARPS[mode, d]))))
    # equal pieces of a run of P pages: ceil(P / ceil(P / length)) pages each
    most = sum(8 * -(-(-(-n // 16)) // shortest) for n in lens)
    assert len(items) <= most
    assert items[:, 1].max() <= 128
