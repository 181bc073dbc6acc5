"""The calls that a user of this library makes, at the sizes they are made at.

The library is the self-attention of a Conformer encoder: batches of utterances, 4 or 8 heads of 64 (d_model 256 or 512),
T positions of 40 ms each after the fourfold down-sampling, bf16 in production and fp32 where a model is checked, usually
with ragged lengths, c = 5 samples per ln T.  `op` says which public call a case times:

  forward   Plan.psattn_forward: steps (a)-(e), the layer that draws its own selection
  reuse     Plan.psattn_forward_with_selection: the N_share - 1 layers that take over another layer's selection
  layer     projections in front, forward, output matrix behind: the whole attention module of one encoder layer
  literal   psattn_forward with the paper's own count, u = r_sparse L, and the query's own value row as the fill
  host      psattn_forward_host: the same path from pinned host buffers to pinned host buffers
"""
import math

import torch

from paper_2106_09236_b200 import binding as ps

D = 64


def _case(name, op, B, H, T, dtype="bf16", c=5.0, shortest=1.0, peaky=0.10, scale=3.0):
    """shortest: the lengths are uniform in [shortest * T, T] (1.0: every sequence is full)."""
    return {"name": name, "op": op, "B": B, "H": H, "T": T, "dtype": dtype, "c": c, "shortest": shortest,
            "peaky": peaky, "scale": scale}


def listed():
    return [
        # the correctness configuration: one 5 s utterance in fp32; nothing but latency
        _case("tiny_fp32", "forward", 1, 4, 128, "fp32"),
        # one 8 s utterance decoded alone, as an interactive service does; an odd length
        _case("utterance_bf16", "forward", 1, 4, 203),
        # the training / batch-scoring shapes of the base and large models
        _case("base_bf16", "forward", 32, 4, 512),
        _case("ragged_bf16", "forward", 64, 4, 500, shortest=0.08),
        _case("large_bf16", "forward", 16, 8, 1024, peaky=0.05, scale=4.0),
        # a few two-minute segments of different lengths: keys no longer fit on chip, odd T
        _case("segments_bf16", "forward", 6, 8, 3001, shortest=0.35),
        # minutes-scale audio
        _case("long_bf16", "forward", 4, 8, 8192),
        # a batch in fp32: a model under validation
        _case("batch_fp32", "forward", 8, 4, 777, "fp32", shortest=0.3),
        # a layer that shares the selection of the layer before it
        _case("reuse_large_bf16", "reuse", 16, 8, 1024, peaky=0.05, scale=4.0),
        # the whole attention module of a layer
        _case("layer_large_bf16", "layer", 16, 8, 1024, shortest=0.5),
        # the setting the paper timed: r_sample = 1, r_sparse = 0.5
        _case("literal_bf16", "literal", 12, 8, 960, c=1.0, shortest=0.4),
        # features that come from and results that go to host memory
        _case("host_base_bf16", "host", 32, 4, 512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# op -> dtype, share of the draws, T range, most rows B * H * T, most B
_RANGES = [
    ("forward", "bf16", 0.50, (64, 8192), 262144, 64),
    ("forward", "fp32", 0.14, (64, 1024), 24864, 16),
    ("reuse", "bf16", 0.10, (64, 8192), 262144, 64),
    ("layer", "bf16", 0.10, (64, 4096), 131072, 64),
    ("literal", "bf16", 0.08, (64, 1536), 92160, 32),
    ("host", "bf16", 0.08, (64, 4096), 65536, 64),
]


def draw(rng):
    x = rng.random()
    for op, dtype, share, (lo, hi), rows, most_b in _RANGES:
        x -= share
        if x < 0:
            break
    T = _log_int(rng, lo, hi)
    H = rng.choice((4, 8))
    B = min(most_b, _log_int(rng, 1, max(1, rows // (H * T))))
    if op == "literal":
        c = 1.0
    else:
        c = 5.0 if rng.random() < 0.75 else round(rng.uniform(2.0, 6.0), 2)
    case = _case("", op, B, H, T, dtype, c, round(rng.choice((1.0, rng.uniform(0.1, 0.9))), 3),
                 *rng.choice(((0.10, 3.0), (0.05, 4.0))))
    del case["name"]
    return case


def _count(c, n):
    return max(1, min(n, math.ceil(c * math.log(n)))) if n > 0 else 0


def _kept(case, n):
    """Number of selected queries of a sequence of n positions."""
    return max(1, min(n, math.ceil(0.5 * n))) if case["op"] == "literal" else _count(case["c"], n)


def _shortest(case):
    return max(1, min(case["T"], int(round(case["shortest"] * case["T"]))))


def _lengths(case, gen):
    lo, T = _shortest(case), case["T"]
    n = torch.randint(lo, T + 1, (case["B"],), generator=gen, device="cuda", dtype=torch.int32)
    n[0] = T                               # a batch is padded to its longest sequence
    return n


def _qkv(case, gen, lengths, dtype):
    """Q, K, V ~ N(0, 1); a share of the queries gets a multiple of one key row added, so that these have the far from
    uniform attention that the measure looks for.  Padded rows are zero."""
    B, H, T = case["B"], case["H"], case["T"]
    q, k, v = (torch.randn((B, H, T, D), generator=gen, device="cuda") for _ in range(3))
    peaky = torch.rand((B, H, T), generator=gen, device="cuda") < case["peaky"]
    key = (torch.rand((B, H, T), generator=gen, device="cuda") * lengths.view(B, 1, 1)).long()
    q += case["scale"] * peaky.unsqueeze(-1) * torch.gather(k, 2, key.unsqueeze(-1).expand(-1, -1, -1, D))
    valid = (torch.arange(T, device="cuda") < lengths.view(B, 1)).view(B, 1, T, 1)
    return [(x * valid).to(dtype) for x in (q, k, v)], peaky & valid.squeeze(-1)


def _samples(case, gen, lengths):
    """Sampled key positions of every query, uniform with replacement over its sequence's valid keys."""
    n = _count(case["c"], case["T"])
    x = torch.rand((case["B"], case["T"], n), generator=gen, device="cuda") * lengths.view(-1, 1, 1)
    return torch.minimum(x.to(torch.int32), lengths.view(-1, 1, 1) - 1).contiguous()


def _selection(case, gen, lengths, peaky, u_max):
    """An index set as an earlier layer would leave it: peaky queries first, ascending, -1 behind the last."""
    B, T = case["B"], case["T"]
    r = torch.rand(peaky.shape, generator=gen, device="cuda") + peaky
    r.masked_fill_((torch.arange(T, device="cuda") >= lengths.view(B, 1)).view(B, 1, T), -1.0)
    at = r.topk(u_max, dim=2).indices.to(torch.int32)
    u = torch.tensor([_kept(case, n) for n in lengths.tolist()], device="cuda").view(B, 1, 1)
    at.masked_fill_(torch.arange(u_max, device="cuda").view(1, 1, -1) >= u, T)
    at = at.sort(dim=2).values
    return at.masked_fill_(at == T, -1).contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    B, H, T, op = case["B"], case["H"], case["T"], case["op"]
    dtype = torch.float32 if case["dtype"] == "fp32" else torch.bfloat16
    lengths = _lengths(case, gen)
    idx = _samples(case, gen, lengths)
    more = {"r_sparse": 0.5, "fill_mode": ps.PSATTN_FILL_OWN_V} if op == "literal" else {}
    plan = ps.Plan(B, H, T, dtype=dtype, c=case["c"], idx_cols=idx.shape[2], **more)
    s = {"op": op, "plan": plan, "lengths": lengths, "idx": idx}
    if op == "layer":
        dx = H * D
        x = torch.randn((B, T, dx), generator=gen, device="cuda")
        s["X"] = (x * (torch.arange(T, device="cuda") < lengths.view(B, 1)).unsqueeze(-1)).to(dtype)
        s["Wt"] = (torch.randn((3, dx, dx), generator=gen, device="cuda") / math.sqrt(dx)).to(dtype)
        s["Wot"] = (torch.randn((dx, dx), generator=gen, device="cuda") / math.sqrt(dx)).to(dtype)
        return s
    (s["Q"], s["K"], s["V"]), peaky = _qkv(case, gen, lengths, dtype)
    if op == "reuse":
        s["sel"] = _selection(case, gen, lengths, peaky, plan.u_max)
        del s["idx"]
    if op == "host":
        for name in ("Q", "K", "V", "lengths", "idx"):
            s[name] = torch.empty(s[name].shape, dtype=s[name].dtype, pin_memory=True).copy_(s[name])
        s["O"] = torch.empty((B, H, T, D), dtype=dtype, pin_memory=True)
        s["sel"] = torch.empty((B, H, plan.u_max), dtype=torch.int32, pin_memory=True)
        plan.psattn_plan_enable_host_io()
    return s


def run(s):
    p, op = s["plan"], s["op"]
    if op == "reuse":
        return p.psattn_forward_with_selection(s["Q"], s["K"], s["V"], s["lengths"], s["sel"])
    if op == "host":
        return p.psattn_forward_host(s["Q"], s["K"], s["V"], s["lengths"], s["idx"], s["O"], s["sel"])
    if op == "layer":
        Q, K, V = p.psattn_project_qkv(s["X"], s["Wt"], s["lengths"])
        O, sel = p.psattn_forward(Q, K, V, s["lengths"], s["idx"])
        return O, sel, p.psattn_project_out(O, sel, s["lengths"], s["Wot"])
    return p.psattn_forward(s["Q"], s["K"], s["V"], s["lengths"], s["idx"])


def work(case):
    """One pass: inputs read once, outputs written once; the products of the sampled scores and of the selected rows'
    attention (and of the projections).  The mean length stands for the lengths."""
    B, H, T, op = case["B"], case["H"], case["T"], case["op"]
    e = 4 if case["dtype"] == "fp32" else 2
    n = (_shortest(case) + T) / 2
    rows, units = B * H * n, B * H
    U, u = _count(case["c"], int(n)), _kept(case, int(n))
    out = B * H * T * D * e
    attend = units * u * n * 4 * D
    score = rows * U * 2 * D
    if op == "reuse":
        return {"bytes": 3 * rows * D * e + out + units * u * 4, "flops": attend}
    path = 3 * rows * D * e + B * n * U * 4 + out + units * u * 4
    if op == "layer":
        dx = H * D
        # X and the weights in, O, the index set and Y out; the output matrix on one fill row and u rows per unit
        return {"bytes": B * n * dx * e + 4 * dx * dx * e + B * n * U * 4 + 2 * out + units * u * 4,
                "flops": B * n * 6.0 * dx * dx + score + attend + units * (u + 1) * 2 * D * dx}
    return {"bytes": path, "flops": score + attend}


def tolerance(case):
    """fp32 sums for fp32 inputs; bf16 weights and results for bf16 inputs.  Index sets: two queries whose measures agree
    to rounding may change places, which moves the entries of that unit."""
    if case["dtype"] == "fp32":
        return {"rel": 1e-5, "max": 4e-4, "differ": 0.01}
    return {"rel": 1e-2, "max": 0.4, "differ": 0.01}
