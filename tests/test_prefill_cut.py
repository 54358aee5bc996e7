"""The cut of a prefill's paths: short chunks under a prefix, whose few rows make
few partials, are cut over the CTAs that would stay idle; a queue that fills the
CTAs with whole paths, or would gain less than its merge costs, stays whole."""
import pytest

from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests.test_prefill_plan import verify_prefill_plan

SMS = 152


def _tree(mode, h_q, h_kv, prefix, chunks, tokens):
    return W.build_prefill("cut", [-1] + [0] * chunks, [prefix] + [tokens] * chunks,
                           list(range(1, chunks + 1)), num_q_heads=h_q, num_kv_heads=h_kv,
                           head_dim=128, mode=mode, values=False)


# pairs of tiles: tokens of a chunk over 2 floor(128 / g), per chunk and kv head
@pytest.mark.parametrize("mode,h_q,h_kv,prefix,chunks,tokens,pairs", [
    ("bf16", 16, 16, 2048, 4, 33, 64),
    ("bf16", 32, 8, 1000, 4, 33, 32),
    ("bf16", 32, 8, 1000, 1, 200, 32),
    ("fp8", 16, 16, 1000, 4, 33, 64),
    ("fp8", 16, 16, 200, 1, 200, 16),
    ("fp8", 28, 4, 200, 1, 64, 8),
])
def test_short_chunks_are_cut(mode, h_q, h_kv, prefix, chunks, tokens, pairs):
    tree = _tree(mode, h_q, h_kv, prefix, chunks, tokens)
    with Plan.for_prefill(tree, host_only=True, num_sms=SMS) as plan:
        verify_prefill_plan(tree, plan)
        entries = plan.info()["num_wide_items"] // 2
        assert entries >= 2 * pairs and entries <= 4 * pairs
        assert plan.launches_per_decode() == 2
        assert plan.workspace_bytes > 0


@pytest.mark.parametrize("mode", ["bf16", "fp8"])
@pytest.mark.parametrize("prefix,chunks,tokens", [(2048, 16, 64), (100, 8, 20), (1, 1, 1)])
def test_whole_paths_stay_whole(mode, prefix, chunks, tokens):
    tree = _tree(mode, 32, 8, prefix, chunks, tokens)
    with Plan.for_prefill(tree, host_only=True, num_sms=SMS) as plan:
        assert plan.launches_per_decode() == 1
        assert plan.workspace_bytes == 0        # the kernel writes the result: no partial rows
