"""Attention of few listed rows over many chunks of keys: one tile of 16 rows leaves more key groups than a chunk has blocks, so a
warp has work in every other chunk only, while the ring of stages goes round several times.  Row counts up to the edge of the tile
(the column-sum row included), CTAs alone on their SM, two per SM, in clusters, and the kernel for row lists."""
import numpy as np
import pytest
import torch

import parity
from oracle import psattn_oracle as orc
from paper_2106_09236_b200 import binding as ps
from paper_2106_09236_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _inputs(B, H, T, c, u, shortest):
    rng = np.random.default_rng(T + B)
    lengths = rng.integers(shortest, T + 1, size=B).astype(np.int32)
    lengths[0] = T
    w = wl.Workload("ring", 0, B, H, T, 64, "bf16", c, 0.1, 3.0)
    n = max(orc.count(c, L) for L in range(1, T + 1))
    inp = wl.make_inputs(w, n, seed=T, lengths=lengths)
    plan = ps.Plan(B, H, T, c=c, idx_cols=n, u_override=u)
    dev = [torch.from_numpy(inp[x]).to("cuda", torch.bfloat16) for x in ("Q", "K", "V")]
    return inp, plan, dev, torch.from_numpy(inp["lengths"]).cuda(), torch.from_numpy(inp["sample_idx"]).cuda()


@pytest.mark.parametrize("B,H,T,c,u,shortest", [
    (75, 1, 3000, 1.0, 0, 3000), (75, 1, 2050, 1.0, 15, 100), (75, 1, 1800, 1.0, 16, 1000), (150, 1, 2600, 1.0, 0, 100),
    (40, 1, 7000, 1.0, 0, 5000), (60, 4, 1400, 1.0, 0, 300), (1, 2, 8600, 1.0, 1, 8600),
])
def test_few_rows_over_many_chunks(B, H, T, c, u, shortest):
    inp, plan, (q, k, v), ln, idx = _inputs(B, H, T, c, u, shortest)
    M = torch.full((B, H, T), float("nan"), device="cuda")
    O, sel = plan.psattn_forward(q, k, v, ln, idx, M_out=M)
    first = O.clone()
    for _ in range(5):
        again, _ = plan.psattn_forward(q, k, v, ln, idx)
        assert torch.equal(again, first)                     # the sums are taken in a fixed order
    given = plan.psattn_forward_with_selection(q, k, v, ln, sel)
    torch.testing.assert_close(given.float(), O.float(), atol=2e-2, rtol=0)
    assert plan.psattn_read_status() == 0
    parity.check_forward(O.float().cpu().numpy(), sel.cpu().numpy(), M.cpu().numpy(), inp, inp["lengths"], "bf16", c, u_override=u)
    plan.close()


@pytest.mark.parametrize("B,T,n_rows", [(150, 2600, 9), (150, 2600, 16), (40, 5000, 3)])
def test_short_row_lists_over_many_chunks(B, T, n_rows):
    inp, plan, (q, k, v), ln, _ = _inputs(B, 1, T, 5.0, 0, T // 2)
    rng = np.random.default_rng(n_rows)
    rows = np.stack([rng.choice(L, size=(1, n_rows), replace=False) for L in inp["lengths"]]).astype(np.int32)
    out = plan.psattn_attend_rows(q, k, v, ln, torch.from_numpy(rows).cuda())
    assert plan.psattn_read_status() == 0
    out = out.cpu().numpy()
    for b in range(0, B, 7):
        for r in range(n_rows):
            ref = orc.attend_row(inp["Q"], inp["K"], inp["V"], b, 0, int(rows[b, 0, r]), int(inp["lengths"][b]))
            assert np.abs(out[b, 0, r] - ref).max() <= 8e-3          # fp32 rows; weights rounded to bf16 meet |V| <= 4
    plan.close()
