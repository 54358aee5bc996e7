"""The prefill kernel at its edges: tiles of one row to a pair of full ones
(32 tokens of 4 q heads are a tile), ancestors that end in every part of a
128-token block, pages in pool order (one box a block) and permuted (a box a
page), whole paths that the kernel finishes itself and paths cut into pieces
that a merge follows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_24658_gb300 import _lib
from paper_2608_24658_gb300 import workloads as W
from paper_2608_24658_gb300.api import Plan
from tests import parity as PT

pytestmark = pytest.mark.gpu


def check(tree, whole=None):
    with Plan.for_prefill(tree) as plan:
        if whole is not None:
            assert plan.launches_per_decode() == (1 if whole else 2)
        out, lse = plan.decode_tree(tree)
        plan.check()
    host = tree.to("cpu")
    kw = oracle.tree_kwargs(host)
    kw["chunk_node"] = kw.pop("leaf_node")
    ref_o, ref_l = oracle.prefill(**kw)
    PT.compare(tree, out, lse, ref_o, ref_l, None, tree.name)


def edges_tree(mode, permute=False):
    prefixes = [1, 63, 64, 65, 127, 128, 129, 300]
    chunks = [1, 31, 32, 33, 63, 64, 65, 2]
    n = len(prefixes)
    return W.build_prefill("edges", [-1] * n + list(range(n)), prefixes + chunks,
                           list(range(n, 2 * n)), num_q_heads=8, num_kv_heads=2, head_dim=128,
                           mode=mode, seed=3, permute_pages=permute, extra_pages=5,
                           tail_value=float("nan"), q_std=0.35, device="cuda")


def fork_tree(mode):
    """9 chunks of 70 tokens, 32 q / 8 kv heads: 144 pairs, every other of 6 tokens."""
    return W.build_prefill("fork", [-1] + [0] * 9, [100] + [70] * 9, list(range(1, 10)),
                           num_q_heads=32, num_kv_heads=8, head_dim=128, mode=mode, seed=8,
                           q_std=0.35, device="cuda")


@pytest.mark.parametrize("permute", [False, True])
@pytest.mark.parametrize("mode", ["bf16", "fp8"])
def test_prefill_tile_and_block_edges(mode, permute):
    tree = edges_tree(mode, permute)
    check(tree)


@pytest.mark.parametrize("mode", ["bf16", "fp8"])
@pytest.mark.parametrize("g", [1, 5, 8, 16])
def test_prefill_cut_paths(mode, g):
    """One chunk over a long chain, more CTAs than pairs: pieces and a merge."""
    tree = W.build_prefill("cut", [-1, 0, 1, 2], [2500, 70, 1337, 40], [3], num_q_heads=g,
                           num_kv_heads=1, head_dim=128, mode=mode, seed=4, q_std=0.35,
                           tail_value=float("nan"), device="cuda")
    check(tree, whole=False)


@pytest.mark.parametrize("mode", ["bf16", "fp8"])
def test_prefill_growing_maxima(mode):
    """Keys that grow along the path move the reference max block after block."""
    tree = W.build_prefill("grow", [-1, 0], [900, 50], [1], num_q_heads=8, num_kv_heads=2,
                           head_dim=128, mode=mode, seed=5, q_std=0.35, device="cuda")
    # (a ramp up to 1, with the growth in the scale of q: e4m3 keys already
    # reach the format's largest value)
    ramp = torch.linspace(0.03, 1.0, tree.k_pages.shape[0], device="cuda").view(-1, 1, 1, 1)
    tree.k_pages.copy_((tree.k_pages.float() * ramp).to(tree.k_pages.dtype))
    tree.q.mul_(3.0)
    check(tree)


@pytest.mark.parametrize("name,mode", [("edges", "bf16"), ("fork", "bf16"), ("fork", "fp8")])
def test_prefill_whole_paths_write_the_result(name, mode):
    """Every pair whole and on a CTA of its own: the attention kernel is the only
    launch.  Several calls on other q, one after the other and one without lse
    (no merge sets the queue counters back between them), each against the
    oracle."""
    tree = edges_tree(mode) if name == "edges" else fork_tree(mode)
    with Plan.for_prefill(tree) as plan:
        assert plan.launches_per_decode() == 1
        mrng = plan.export(_lib.TABLE_MERGE_RANGES)
        assert (mrng[:, 1] - mrng[:, 0] == 1).all()
        q0, got = tree.q.clone(), []
        for k, want_lse in enumerate((True, False, True)):
            tree.q.copy_(q0.roll(k, dims=0))
            got.append(plan.decode_tree(tree, want_lse=want_lse))
        plan.check()
    assert got[1][1] is None
    for k, (out, lse) in enumerate(got):
        tree.q.copy_(q0.roll(k, dims=0))
        kw = oracle.tree_kwargs(tree.to("cpu"))
        kw["chunk_node"] = kw.pop("leaf_node")
        ref_o, ref_l = oracle.prefill(**kw)
        PT.compare(tree, out, lse, ref_o, ref_l, None, f"{tree.name} call {k}")


@pytest.mark.parametrize("mode", ["bf16", "fp8"])
def test_prefill_whole_paths_need_no_workspace(mode):
    tree = fork_tree(mode)
    with Plan.for_prefill(tree) as plan:
        assert plan.workspace_bytes == 0
        ref = plan.decode_tree(tree)
        out, lse = torch.full_like(tree.q, float("nan")), torch.full_like(ref[1], float("nan"))
        scales = [None if s is None else s.data_ptr() for s in (tree.k_scale, tree.v_scale)]
        st = _lib.load().parason_attn_decode(
            plan.handle, tree.q.data_ptr(), tree.k_pages.data_ptr(), tree.v_pages.data_ptr(), *scales,
            out.data_ptr(), lse.data_ptr(), None, 0, torch.cuda.current_stream().cuda_stream)
        plan.check()
        assert st == 0 and torch.equal(out, ref[0]) and torch.equal(lse, ref[1])
        out.fill_(float("nan"))
        plan.decode_no_alloc(tree.q, tree.k_pages, tree.v_pages, out, lse, k_scale=tree.k_scale,
                             v_scale=tree.v_scale)
        plan.check()
        assert torch.equal(out, ref[0])


def test_prefill_e4m3_many_pairs():
    """More than 4 tile pairs per SM with e4m3 KV: several whole paths a CTA, and a merge."""
    n = 4 * torch.cuda.get_device_properties(0).multi_processor_count // 16 + 2
    tree = W.build_prefill("many", [-1, 0] + [1] * n, [70, 9] + [1 + k % 3 for k in range(n)],
                           list(range(2, 2 + n)), num_q_heads=16, num_kv_heads=16, head_dim=128,
                           mode="fp8", seed=6, q_std=0.35, tail_value=float("nan"), device="cuda")
    check(tree, whole=False)
