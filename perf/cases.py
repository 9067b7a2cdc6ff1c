"""Performance cases of the gated-delta-rule library: the calls that a training program makes, over the range of sizes,
data types and gate settings that the entry points take.

A case is one mixer layer of one training step.  `entry` is "bwd" (the gradients alone, everything recomputed: activation
checkpointing) or "step" (forward with its output, then the backward on the workspace the forward left).  `gates` is
"scalar" (one log decay and one beta per token and head: gdn_fwd_recompute / gdn_bwd) or the family member of the calls
with per-channel gates ("kda": one beta for both gates, "gla": erase 0 and write 1, "gdn": three independent vectors).
Values are drawn as in the library's synthetic workloads: unit q and k, normal v and dO, beta = sigmoid(normal),
log decay = -decay * softplus(normal), states normal with deviation 0.1 (given, or absent)."""
import math

import torch
import torch.nn.functional as F

from paper_2608_12700_b200 import binding

CHUNK = 64


def _case(name, entry, gates, dtype, seqs, tokens, heads, d_k, d_v, packed=False, states=False, delta=1, decay=0.1):
    """`tokens`: of each sequence, or with `packed` of all sequences together."""
    return dict(name=name, entry=entry, gates=gates, dtype=dtype, seqs=seqs, tokens=tokens, heads=heads, d_k=d_k, d_v=d_v,
                packed=packed, states=states, delta=delta, decay=decay)


def listed():
    return [
        # the smallest fp32 call: a unit-sized layer, as in gradient checks and toy models; all launches and latency
        _case("f32_smallest", "bwd", "scalar", "f32", 1, 128, 2, 64, 64),
        # a short odd-length sequence in bf16: fine-tuning on single short documents, one training step
        _case("bf16_short_step", "step", "scalar", "bf16", 1, 333, 4, 128, 128),
        # the ordinary training shape: gradients of one layer, recomputed (activation checkpointing)
        _case("bf16_train", "bwd", "scalar", "bf16", 4, 2048, 16, 128, 128, states=True),
        # the same layer without checkpointing (forward, then backward on its workspace), lengths that end in a short chunk
        _case("bf16_ragged_step", "step", "scalar", "bf16", 6, 1500, 16, 128, 128),
        # one long document: few chains, many chunks
        _case("bf16_long", "bwd", "scalar", "bf16", 1, 16384, 16, 128, 128, states=True),
        # packed documents of uneven lengths, the largest call
        _case("bf16_packed", "bwd", "scalar", "bf16", 8, 32768, 32, 128, 128, packed=True, states=True),
        # the scalar-gate recurrence without the delta rule (SSD-like), narrow heads
        _case("bf16_ssd", "bwd", "scalar", "bf16", 8, 4096, 32, 64, 64, delta=0, decay=0.05),
        # value heads half as wide as the key heads
        _case("bf16_narrow_values", "step", "scalar", "bf16", 4, 2048, 16, 128, 64),
        # fp32 training step of a small layer with an odd length
        _case("f32_step", "step", "scalar", "f32", 2, 1000, 4, 128, 128, states=True),
        # per-channel decay (KDA), the ordinary training shape
        _case("kda_train", "bwd", "kda", "bf16", 4, 2048, 16, 128, 128, states=True),
        # per-channel gates in fp32: a small layer, one training step, three independent gate vectors
        _case("channelwise_f32_step", "step", "gdn", "f32", 2, 500, 4, 64, 64),
        # per-channel decay so fast that a chunk's cumulative factor underflows (channels that forget within a few tokens)
        _case("kda_fast_decay", "bwd", "kda", "bf16", 1, 1024, 8, 128, 128, decay=4.0),
    ]


# What drawn cases vary over, one row for each listed kind: (entry, gates, dtype, delta rule, pairs of head dimensions,
# decays, largest number of tokens times heads, most tokens of one sequence).  The bounds keep a drawn call below the
# largest listed one in time.
_WIDE = ((128, 128),)
_ANY = ((128, 128), (128, 64), (64, 128), (64, 64))
_KINDS = (
    ("bwd", "scalar", "bf16", 1, _WIDE, (0.05, 0.1, 0.3), 900000, 16384),
    ("step", "scalar", "bf16", 1, _WIDE, (0.05, 0.1, 0.3), 700000, 16384),
    ("bwd", "scalar", "bf16", 1, ((128, 64), (64, 128), (64, 64)), (0.05, 0.1), 300000, 8192),
    ("step", "scalar", "bf16", 1, ((128, 64),), (0.05, 0.1), 300000, 8192),
    ("bwd", "scalar", "bf16", 0, ((64, 64), (64, 64), (128, 128)), (0.05, 0.1), 600000, 8192),
    ("bwd", "scalar", "f32", 1, _ANY, (0.05, 0.1), 6000, 600),
    ("step", "scalar", "f32", 1, _ANY, (0.05, 0.1), 6000, 600),
    ("bwd", "kda", "bf16", 1, ((128, 128), (128, 128), (128, 64)), (0.05, 0.1), 150000, 8192),
    ("step", "gla", "bf16", 1, _WIDE, (0.05, 0.1), 150000, 8192),
    ("step", "gdn", "f32", 1, ((64, 64), (128, 128)), (0.05, 0.1), 3000, 400),
    ("bwd", "kda", "bf16", 1, _WIDE, (3.0, 4.0), 5000, 800),
)


def draw(rng):
    entry, gates, dtype, delta, dims, decays, most, longest = rng.choice(_KINDS)
    d_k, d_v = rng.choice(dims)
    work = math.exp(rng.uniform(math.log(256.0), math.log(most)))          # tokens times heads
    heads = min(rng.choice((1, 2, 4, 6, 8, 16, 24, 32)), max(1, int(work) // 96))
    tokens = max(33, int(work / heads))                                    # of the whole batch
    seqs = max(-(-tokens // longest), min(rng.choice((1, 1, 2, 3, 4, 8, 12)), max(1, tokens // 48)))
    packed = rng.random() < 0.3
    per_row = tokens // seqs
    if rng.random() < 0.4 and per_row >= 64:                               # whole chunks as often as odd lengths
        per_row -= per_row % 64
    case = _case(None, entry, gates, dtype, seqs, per_row * seqs if packed else per_row, heads, d_k, d_v, packed=packed,
                 states=rng.random() < 0.5, delta=delta, decay=rng.choice(decays))
    del case["name"]
    return case


def _sizes(case):
    rows = 1 if case["packed"] else case["seqs"]
    return rows, case["tokens"], rows * case["tokens"]


def _lengths(case, gen):
    """Uneven lengths of the packed sequences: a share of the tokens each, between a quarter and the whole of one weight."""
    w = 0.25 + 0.75 * torch.rand(case["seqs"], generator=gen, dtype=torch.float64)
    cut = (torch.cumsum(w, 0) / w.sum() * case["tokens"]).round().to(torch.int32)
    cut[-1] = case["tokens"]
    return torch.cat([torch.zeros(1, dtype=torch.int32), cut])


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rows, T, total = _sizes(case)
    H, dk, dv, N = case["heads"], case["d_k"], case["d_v"], case["seqs"]
    io = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    vec = case["gates"] != "scalar"

    def normal(*shape):
        return torch.randn(shape, generator=gen, device=dev)

    def new(*shape, dtype=torch.float32):
        return torch.empty(shape, dtype=dtype, device=dev)

    s = dict(case=case)
    s["q"], s["k"] = (F.normalize(normal(rows, T, H, dk), dim=-1).to(io) for _ in range(2))
    s["v"], s["dO"] = (normal(rows, T, H, dv).to(io) for _ in range(2))
    decay_shape = (rows, T, H, dk) if vec else (rows, T, H)
    s["g"] = -case["decay"] * F.softplus(normal(*decay_shape))
    if case["gates"] == "scalar":
        s["beta"] = torch.sigmoid(normal(rows, T, H)) if case["delta"] else None
    elif case["gates"] == "kda":
        beta = torch.sigmoid(normal(rows, T, H, 1))
        s["b"], s["w"] = beta.expand(rows, T, H, dk).contiguous(), beta.expand(rows, T, H, dv).contiguous()
    elif case["gates"] == "gla":
        s["b"], s["w"] = torch.zeros_like(s["g"]), torch.ones((rows, T, H, dv), device=dev)
    else:
        s["b"], s["w"] = torch.sigmoid(normal(rows, T, H, dk)), torch.sigmoid(normal(rows, T, H, dv))
    s["h0"], s["dhT"] = ((0.1 * normal(N, H, dk, dv)) for _ in range(2)) if case["states"] else (None, None)
    s["cu"] = None
    if case["packed"]:
        host = torch.Generator()
        host.manual_seed(seed)
        s["cu"] = _lengths(case, host).to(dev)

    s["desc"] = binding.make_desc(B=rows, T=T, H=H, d_k=dk, d_v=dv, N=N, dtype=case["dtype"], delta_rule=case["delta"])
    size = binding.gdn_workspace_bytes_channelwise if vec else binding.gdn_workspace_bytes
    s["ws"] = new(size(s["desc"])[1], dtype=torch.uint8)
    out = dict(dq=new(rows, T, H, dk, dtype=io), dk=new(rows, T, H, dk, dtype=io), dv=new(rows, T, H, dv, dtype=io),
               dg=new(*decay_shape))
    if vec:
        out["db"], out["dw"] = new(rows, T, H, dk), new(rows, T, H, dv)
    elif case["delta"]:
        out["dbeta"] = new(rows, T, H)
    if case["states"]:
        out["dh0"] = new(N, H, dk, dv)
    if case["entry"] == "step":
        out["o"] = new(rows, T, H, dv, dtype=io)
        if case["states"]:
            out["hT"] = new(N, H, dk, dv)
    s["out"] = out
    return s


def run(s):
    case, out = s["case"], s["out"]
    step = case["entry"] == "step"
    tensors = (s["desc"], s["q"], s["k"], s["v"], s["g"])
    if case["gates"] == "scalar":
        gates = (s["beta"],)
        fwd, bwd, gate_grads = binding.gdn_fwd_recompute, binding.gdn_bwd, (out.get("dbeta"),)
    else:
        gates = (s["b"], s["w"])
        fwd, bwd, gate_grads = binding.gdn_fwd_recompute_channelwise, binding.gdn_bwd_channelwise, (out["db"], out["dw"])
    if step:
        fwd(*tensors, *gates, s["h0"], s["cu"], out["o"], out.get("hT"), s["ws"])
    bwd(*tensors, *gates, s["h0"], s["dO"], s["dhT"], s["cu"], out["dq"], out["dk"], out["dv"], out["dg"], *gate_grads,
        out.get("dh0"), s["ws"], workspace_is_fresh_from_fwd=int(step))
    return out


def work(case):
    """Inputs read once and outputs written once (a step reads q, k, v and the gates in the forward and again, with dO, in
    the backward); products of the chunkwise method, a triangular one at half."""
    _, _, total = _sizes(case)
    dk, dv, H = case["d_k"], case["d_v"], case["heads"]
    io = 2 if case["dtype"] == "bf16" else 4
    if case["gates"] == "scalar":
        gates = 4 * (1 + case["delta"])
    else:
        gates = 4 * (2 * dk + dv)
    inputs, outputs = (2 * dk + dv) * io + gates, (2 * dk + dv) * io + gates
    n_bytes = total * H * (inputs + dv * io + outputs)
    chains, state = case["seqs"] * H, 4 * dk * dv
    if case["states"]:
        n_bytes += 3 * chains * state
    tri_k, tri_v, dense = CHUNK * dk, CHUNK * dv, 2 * dk * dv              # flops of one token
    if case["delta"] or case["gates"] != "scalar":
        flops = 9 * tri_k + 5 * tri_v + 8 * dense + 2 * CHUNK ** 2 // 3
    else:
        flops = 3 * tri_k + 2 * tri_v + 5 * dense
    if case["entry"] == "step":
        n_bytes += total * H * (inputs + dv * io) + (2 * chains * state if case["states"] else 0)
        flops += tri_v + dense                                             # the output: P U and Q h
    return {"bytes": n_bytes, "flops": total * H * flops}


def tolerance(case):
    # Errors against the float64 oracle over the listed cases, times four.  bf16 (every operand of a product is rounded):
    # 3.7e-3, largest entry 0.037 of the root mean square, with scalar gates; 6.6e-3 (the decay gradient) and 0.11 with
    # per-channel gates.  fp32: 6.4e-7 and 4.3e-6.
    if case["dtype"] == "f32":
        return {"rel": 2.6e-6, "max": 2e-5}
    return {"rel": 1.5e-2, "max": 0.15} if case["gates"] == "scalar" else {"rel": 2.6e-2, "max": 0.45}
