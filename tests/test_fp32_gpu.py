"""fp32 mode on the GPU at the edges of its kernel: every split of a tile's
rows over warps (1 to 16 rows, full and partial row groups), pieces of one
page to more than a ring, last pages of one token and of a whole page."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan

from tests import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("h_q,h_kv", [(2, 2), (3, 1), (8, 2), (5, 1), (8, 1), (9, 1), (12, 1), (16, 1)])
def test_fp32_tile_edges(h_q, h_kv, d):
    lens = [1, 16, 17, 33, 64, 65, 144, 272, 527, 530]
    tree = W.build_tree("fp32_edges", [-1] + [0] * len(lens), [75] + lens,
                        list(range(1, len(lens) + 1)), num_q_heads=h_q, num_kv_heads=h_kv,
                        head_dim=d, mode="fp32", seed=5, permute_pages=True, extra_pages=2,
                        tail_value=float("nan"), device="cuda")
    with Plan.for_tree(tree) as plan:
        out, lse = plan.decode_tree(tree)
        plan.check()
    ref_o, ref_l = oracle.decode(**oracle.tree_kwargs(tree.to("cpu")))
    # every sum is fp32: the mode's stated bounds
    assert np.abs(out.double().cpu().numpy() - ref_o).max() <= parity.FP32_MAX_ABS
    assert np.abs(lse.double().cpu().numpy() - ref_l).max() <= parity.LSE_ABS["fp32"]


def test_fp32_growing_maxima():
    """Scores that grow along the node move the reference max again and again."""
    tree = W.build_tree("fp32_grow", [-1, 0, 0], [600, 40, 7], [1, 2], num_q_heads=8,
                        num_kv_heads=2, head_dim=128, mode="fp32", seed=6, device="cuda")
    tree.k_pages.mul_(torch.linspace(0.1, 4.0, tree.k_pages.shape[0], device="cuda").view(-1, 1, 1, 1))
    with Plan.for_tree(tree) as plan:
        out, lse = plan.decode_tree(tree)
        plan.check()
    ref_o, ref_l = oracle.decode(**oracle.tree_kwargs(tree.to("cpu")))
    # scores reach about 60: an fp32 score's rounding (2^-24 of it, over
    # 128 products) scales p by up to 1 + 60 * 2^-21
    assert np.abs(out.double().cpu().numpy() - ref_o).max() <= 4e-5 * max(1.0, np.abs(ref_o).max())
    assert np.abs(lse.double().cpu().numpy() - ref_l).max() <= 4e-5
