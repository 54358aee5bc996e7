"""parason_lse_merge around the edges of its launch: a row, a partial CTA, and
both sides of the row count at which a lane takes several rows; in place too."""
import math
import os
import re

import pytest
import torch

from paper_2608_24658_gb300.api import lse_merge

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_24658_gb300", "csrc")


def _constant(name):
    with open(os.path.join(CSRC, "merge.cu")) as f:
        return int(re.search(rf"constexpr \w+ {name} = (\d+);", f.read()).group(1))


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("in_place", [False, True])
def test_lse_merge_row_edges(d, dtype, in_place):
    rows_per_pass = _constant("kLseThreads") * 16 // (d * dtype.itemsize)
    wide = _constant("kLseRows") * _constant("kLseWideCtas") * rows_per_pass
    for rows in (1, 3, rows_per_pass, rows_per_pass + 1, wide - 1, wide, wide + 5):
        gen = torch.Generator(device="cuda")
        gen.manual_seed(rows)
        o = [torch.randn((rows, d), generator=gen, device="cuda").to(dtype) for _ in range(2)]
        lse = [3.0 * torch.randn(rows, generator=gen, device="cuda") for _ in range(2)]
        lse[0][::3] = -math.inf
        lse[1][::5] = -math.inf
        la, lb = (x.double() for x in lse)
        ref_l = torch.logaddexp(la, lb)
        wa, wb = (torch.exp(x - ref_l).nan_to_num(0.0)[:, None] for x in (la, lb))
        ref_o = wa * o[0].double() + wb * o[1].double()
        kw = dict(o_out=o[0], lse_out=lse[0]) if in_place else {}
        out, out_l = lse_merge(o[0], lse[0], o[1], lse[1], **kw)
        # one rounding to the output type, beside a few of fp32
        eps = 2.0 ** -8 if dtype == torch.bfloat16 else 2.0 ** -20
        assert ((out.double() - ref_o).abs() <= eps * ref_o.abs() + 2.0 ** -20).all()
        live = ref_l > -math.inf
        assert ((out_l.double() - ref_l)[live].abs() <= 2.0 ** -20 * (1.0 + ref_l[live].abs())).all()
        assert (out_l[~live] == -math.inf).all()
