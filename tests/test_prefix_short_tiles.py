"""A short shared prefix under many branches: its tiles are starts more than
pages, and get CTAs for them; long ones keep the share that their pages give."""
import pytest

from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests.test_plan import verify_plan


def _tree(mode, d, requests, prefix, trials, tokens, **kw):
    parent, lens, leaves = [], [], []
    for _ in range(requests):
        root = len(parent)
        parent.append(-1)
        lens.append(prefix)
        for k in range(trials):
            leaves.append(len(parent))
            parent.append(root)
            lens.append(tokens + k % 7)
    return W.build_tree("short_tiles", parent, lens, leaves, num_q_heads=64, num_kv_heads=8,
                        head_dim=d, mode=mode, seed=3, **kw)


@pytest.mark.parametrize("mode,d", [("bf16", 64), ("bf16", 128), ("fp8", 128)])
@pytest.mark.parametrize("requests,prefix,trials,tokens,least", [
    (1, 1, 64, 500, 8), (1, 64, 64, 500, 8), (8, 64, 32, 200, 16), (16, 16, 20, 2000, 4)])
def test_short_tiles_get_ctas(mode, d, requests, prefix, trials, tokens, least):
    tree = _tree(mode, d, requests, prefix, trials, tokens, values=False)
    with Plan.for_tree(tree, host_only=True, num_sms=152) as plan:
        verify_plan(tree, plan)
        info = plan.info()
    assert least <= info["num_wide_ctas"] <= info["num_wide_items"]
    assert info["num_ctas"] == 152


@pytest.mark.parametrize("sms", [1, 2, 3])
def test_short_tiles_on_few_sms(sms):
    tree = _tree("bf16", 64, 2, 1, 20, 40, values=False)
    with Plan.for_tree(tree, host_only=True, num_sms=sms) as plan:
        verify_plan(tree, plan)
        assert 1 <= plan.info()["num_wide_ctas"] <= max(1, sms - 1)


@pytest.mark.gpu
@pytest.mark.parametrize("mode,d", [("bf16", 64), ("bf16", 128), ("fp8", 128)])
@pytest.mark.parametrize("requests,prefix,trials,tokens", [(1, 1, 64, 40), (16, 16, 20, 60), (8, 64, 9, 1)])
def test_short_tiles_match_the_oracle(mode, d, requests, prefix, trials, tokens):
    from tests import parity
    parity.run_and_compare(_tree(mode, d, requests, prefix, trials, tokens, device="cuda",
                                 permute_pages=True, tail_value=float("nan")))
