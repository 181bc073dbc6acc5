"""More units than SMs (two CTAs of 256 threads per SM): key-tile and row-tile edges, all modes, against the oracle."""
import numpy as np
import pytest
import torch

import parity
from kernels import launched
from oracle import psattn_oracle as orc
from paper_2106_09236_b200 import binding as ps
from paper_2106_09236_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,T,shortest,c,fill", [
    (40, 4, 64, 0, 5.0, 0), (40, 4, 129, 1, 5.0, 1), (75, 4, 200, 200, 5.0, 0), (75, 4, 400, 0, 9.0, 0), (75, 4, 500, 250, 2.0, 0),
    (150, 1, 208, 1, 10.0, 0), (38, 4, 1300, 900, 5.0, 0), (150, 1, 2600, 100, 1.0, 0), (300, 1, 16, 0, 5.0, 0),
    (60, 4, 1150, 1150, 5.0, 0), (60, 4, 1536, 0, 1.0, 0),
])
def test_two_ctas_per_sm(B, H, T, shortest, c, fill):
    rng = np.random.default_rng(T)
    lengths = rng.integers(shortest, T + 1, size=B).astype(np.int32)
    lengths[0] = T
    w = wl.Workload("half", 0, B, H, T, 64, "bf16", c, 0.1, 3.0)
    n = max(orc.count(c, L) for L in range(1, T + 1))
    inp = wl.make_inputs(w, n, seed=T, lengths=lengths, pad_value=float("nan"))
    plan = ps.Plan(B, H, T, c=c, idx_cols=n, fill_mode=fill)
    q, k, v = (torch.from_numpy(inp[x]).to("cuda", torch.bfloat16) for x in ("Q", "K", "V"))
    ln, idx = (torch.from_numpy(inp[x]).cuda() for x in ("lengths", "sample_idx"))
    M = torch.full((B, H, T), float("nan"), device="cuda")
    O, sel = plan.psattn_forward(q, k, v, ln, idx, M_out=M)
    again = plan.psattn_forward_with_selection(q, k, v, ln, sel)
    torch.testing.assert_close(again.float(), O.float(), atol=2e-2, rtol=0)
    assert plan.psattn_read_status() == 0
    plan.close()
    if fill == 0:
        for x in ("Q", "K", "V"):
            inp[x] = np.nan_to_num(inp[x])
        parity.check_forward(O.float().cpu().numpy(), sel.cpu().numpy(), M.cpu().numpy(), inp, inp["lengths"], "bf16", c)
    else:
        staged = ps.Plan(B, H, T, c=c, idx_cols=n, fill_mode=fill, path=ps.PSATTN_PATH_STAGED)
        O2, sel2 = staged.psattn_forward(q, k, v, ln, idx)
        same = (sel2 == sel).all(dim=2)
        assert same.float().mean() > 0.9
        torch.testing.assert_close(O[same].float(), O2[same].float(), atol=2e-2, rtol=0)
        staged.close()


@pytest.mark.parametrize("B,H,T,mode,half", [
    (37, 4, 300, 0, False), (38, 4, 208, 0, True), (38, 4, 209, 0, False), (60, 4, 400, 0, True), (75, 4, 500, 0, True),
    (37, 4, 300, 2, False), (38, 4, 1024, 2, True), (38, 4, 1025, 2, False), (50, 4, 1536, 2, True), (75, 4, 1537, 2, False), (112, 4, 1600, 2, True),
    (58, 4, 1152, 1, False), (60, 4, 1536, 1, True), (75, 4, 1537, 1, False), (112, 4, 1600, 1, True), (112, 4, 4033, 1, False),
])
def test_shape_of_the_ctas_by_size(B, H, T, mode, half):
    """Which of the two shapes a call takes (mode 0: all steps, 1: behind a measure kernel, 2: an index set given)."""
    plan = ps.Plan(B, H, T, c=5.0)
    x = torch.zeros((B, H, T, 64), dtype=torch.bfloat16, device="cuda")
    idx = torch.zeros((B, T, plan.idx_cols), dtype=torch.int32, device="cuda")
    sel = torch.zeros((B, H, plan.u_max), dtype=torch.int32, device="cuda")
    _, ran = launched(lambda: plan.psattn_forward_with_selection(x, x, x, None, sel) if mode == 2 else plan.psattn_forward(x, x, x, None, idx))
    shape = "256,128,2" if half else "512,256,3"
    assert {k for k in ran if k.startswith("k_forward_fused")} == {"k_forward_fused<0,%d,%s>" % (mode, shape)}
    plan.close()
