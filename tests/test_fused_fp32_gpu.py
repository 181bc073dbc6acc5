"""fp32 inputs in one launch: keys resident in shared memory or not, one or several CTAs per unit, chunk and range edges, both fills,
an index set given; against the one-kernel-per-step schedule and the oracle."""
import numpy as np
import pytest
import torch

import parity
from oracle import psattn_oracle as orc
from paper_2106_09236_b200 import binding as ps
from paper_2106_09236_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,lengths,c,fill", [
    (1, 1, [1], 5.0, 0), (4, 95, [95, 1, 64], 5.0, 0), (2, 96, [96, 0, 31], 5.0, 0), (4, 129, [129, 128, 127], 2.0, 1),
    (1, 900, [900], 5.0, 0), (8, 777, [777, 300, 5, 640], 6.0, 0), (4, 1025, [1025, 1, 257], 5.0, 1), (8, 1536, [1536, 1000], 8.0, 0),
    (16, 200, [200, 17, 199, 64, 3, 111, 150, 200, 90, 31, 8], 5.0, 0),
])
def test_fp32_in_one_launch(H, T, lengths, c, fill):
    B = len(lengths)
    w = wl.Workload("f32", 0, B, H, T, 64, "fp32", c, 0.1, 3.0)
    n = max(orc.count(c, L) for L in range(1, T + 1))
    inp = wl.make_inputs(w, n, seed=T, lengths=lengths, pad_value=float("nan"))
    q, k, v = (torch.from_numpy(inp[x]).cuda() for x in ("Q", "K", "V"))
    ln, idx = (torch.from_numpy(inp[x]).cuda() for x in ("lengths", "sample_idx"))
    res = {}
    for path in (ps.PSATTN_PATH_AUTO, ps.PSATTN_PATH_STAGED):
        plan = ps.Plan(B, H, T, dtype=torch.float32, c=c, idx_cols=n, fill_mode=fill, path=path)
        M = torch.full((B, H, T), float("nan"), device="cuda")
        before = ps.psattn_launch_count()
        O, sel = plan.psattn_forward(q, k, v, ln, idx, M_out=M)
        assert (ps.psattn_launch_count() - before == 1) == (path == ps.PSATTN_PATH_AUTO)
        again = plan.psattn_forward_with_selection(q, k, v, ln, sel)
        assert plan.psattn_read_status() == 0
        torch.testing.assert_close(again, O, atol=1e-5, rtol=1e-5)
        res[path] = [x.cpu() for x in (O, sel, M)]
        plan.close()
    (O, sel, M), (O2, sel2, M2) = res[ps.PSATTN_PATH_AUTO], res[ps.PSATTN_PATH_STAGED]
    torch.testing.assert_close(M, M2, atol=1e-5, rtol=1e-5)
    assert torch.equal(sel, sel2)
    torch.testing.assert_close(O, O2, atol=1e-5, rtol=1e-5)
    if fill == 0:
        for x in ("Q", "K", "V"):
            inp[x] = np.nan_to_num(inp[x])
        parity.check_forward(O.numpy(), sel.numpy(), M.numpy(), inp, inp["lengths"], "fp32", c)
