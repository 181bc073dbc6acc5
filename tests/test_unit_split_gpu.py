"""Several CTAs per (batch, head) unit (few units): the ranges of queries, keys and rows that the CTAs of a cluster share out,
at lengths that leave some of them empty, at tile edges, and with an index set given."""
import numpy as np
import pytest
import torch

import parity
from oracle import psattn_oracle as orc
from paper_2106_09236_b200 import binding as ps
from paper_2106_09236_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,lengths,c", [
    (4, 192, [192], 5.0), (2, 193, [1, 193, 8], 5.0), (1, 257, [129, 0, 257], 5.0), (4, 1024, [1024], 5.0),
    (3, 1000, [999, 127, 128, 1000, 65], 3.0), (8, 777, [777, 300, 5, 640], 5.0), (8, 513, [513, 512, 40, 1, 257], 5.0),
    (8, 1024, [1024, 1, 900, 33, 1024, 511, 769, 1000, 2], 5.0),
])
def test_units_shared_by_several_ctas(H, T, lengths, c):
    w = wl.Workload("split", 0, len(lengths), H, T, 64, "bf16", c, 0.1, 3.0)
    n = max(orc.count(c, L) for L in range(1, T + 1))
    inp = wl.make_inputs(w, n, seed=T, lengths=lengths, pad_value=float("nan"))
    plan = ps.Plan(len(lengths), H, T, c=c, idx_cols=n)
    q, k, v = (torch.from_numpy(inp[x]).to("cuda", torch.bfloat16) for x in ("Q", "K", "V"))
    ln, idx = (torch.from_numpy(inp[x]).cuda() for x in ("lengths", "sample_idx"))
    M = torch.full((len(lengths), H, T), float("nan"), device="cuda")
    O, sel = plan.psattn_forward(q, k, v, ln, idx, M_out=M)
    for x in ("Q", "K", "V"):
        inp[x] = np.nan_to_num(inp[x])
    parity.check_forward(O.float().cpu().numpy(), sel.cpu().numpy(), M.cpu().numpy(), inp, inp["lengths"], "bf16", c)
    again = plan.psattn_forward_with_selection(q, k, v, ln, sel)
    torch.testing.assert_close(again.float(), O.float(), atol=2e-2, rtol=0)
    assert plan.psattn_read_status() == 0
    plan.close()
