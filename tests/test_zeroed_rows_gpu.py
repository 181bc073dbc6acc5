"""Projections and output matrix without given outputs: the padded rows of the fresh tensors are zero, whatever the allocator hands
out, at the edges of the 128-token tiles and of the ranges of positions."""
import numpy as np
import pytest
import torch

from oracle import psattn_oracle as orc
from paper_2106_09236_b200 import binding as ps
from paper_2106_09236_b200 import workloads as wl

pytestmark = pytest.mark.gpu


def _poison(n_bytes):
    """Leaves NaN patterns in the allocator's cache for the next tensors of this size."""
    t = torch.full((n_bytes // 4,), float("nan"), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    del t


@pytest.mark.parametrize("dtype,T,lengths", [
    ("bf16", 257, [257, 128, 129, 0, 1]), ("bf16", 130, [130, 127, 0]), ("bf16", 700, [3, 256, 511, 700]), ("fp32", 70, [70, 1, 0]),
])
def test_padded_rows_of_fresh_outputs_are_zero(dtype, T, lengths):
    H, B, dx = 2, len(lengths), 128
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    w = wl.Workload("zeroed", 0, B, H, T, 64, dtype, 2.0, 0.1, 3.0)
    pin = wl.make_projection_inputs(w, lengths=lengths, pad_value=float("nan"))
    plan = ps.Plan(B, H, T, dtype=tdt, c=2.0)
    X, Wt = (torch.from_numpy(pin[k]).to("cuda", tdt) for k in ("X", "Wt"))
    ln = torch.tensor(lengths, dtype=torch.int32, device="cuda")
    n = B * H * T * 64 * X.element_size()
    for _ in range(3):
        _poison(n)
    Q, K, V = plan.psattn_project_qkv(X, Wt, ln)
    ref = orc.project_qkv(np.nan_to_num(pin["X"]), pin["Wt"], H, pin["lengths"], nthreads=2)
    for got, want in zip((Q, K, V), ref):
        got = got.float().cpu().numpy()
        for b, L in enumerate(lengths):
            assert (got[b, :, L:] == 0).all() and np.abs(got[b, :, :L] - want[b, :, :L]).max(initial=0) < 3e-2
    rng = np.random.default_rng(3)
    idx = torch.zeros((B, T, plan.idx_cols), dtype=torch.int32, device="cuda")
    O, sel = plan.psattn_forward(Q, K, V, ln, idx)
    # width 64: the dense product with and without an index set; width 72: the corrections, and one thread per element
    for dy, s in ((64, sel), (64, None), (72, sel), (72, None)):
        Wot = torch.from_numpy((rng.standard_normal((dy, H * 64)) / 11).astype(np.float32)).to("cuda", tdt)
        for _ in range(3):
            _poison(B * T * dy * X.element_size())
        Y = plan.psattn_project_out(O, s, ln, Wot).float().cpu().numpy()
        want = orc.project_out(O.float().cpu().numpy(), Wot.float().cpu().numpy(), pin["lengths"], nthreads=2)
        for b, L in enumerate(lengths):
            assert (Y[b, L:] == 0).all() and np.abs(Y[b, :L] - want[b, :L]).max(initial=0) < 3e-2
    plan.close()
