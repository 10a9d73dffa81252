"""Performance cases of the SwiLA recurrence: what its users call, over the sizes they call it with.

A case is a dict of plain values; ``prepare`` makes what a program has in hand before the call, ``run`` is one pass
through the public entry points of ``paper_2609_39034_b200.binding``.  Kinds:

  decode   one generated token on a carried state, updated in place (generation, App. D.4)
  prefill  a whole sequence from the initial state: prompts of a server, the forward pass of training; with ``stats`` the
           sums behind the load-balancing loss are formed too (Sec. 3.5)
  layer    a prefill on raw q, k, v projections (SiLU and L2 norm inside the kernel) and the output RMSNorm behind it:
           the layer as the paper's models run it (App. B.2, App. D.1)
  host     a prefill whose tensors live in pinned host memory

Values: q and k are SiLU + L2-normalised Gaussians, v SiLU of Gaussians, the gate logits have standard deviation 0.9 (what
the language-model configuration's embedding projections give), decays are sigmoid(3 + Gaussian)."""
import math

import torch

from paper_2609_39034_b200 import binding, workloads as wl

GRANULARITY = {"none": wl.GRAN_NONE, "key": wl.GRAN_PER_KEY, "out": wl.GRAN_PER_OUT, "component": wl.GRAN_SCALAR}
VALUES = ("q", "k", "v", "beta_logit", "pik_logit", "piq_logit", "gk_logit", "gq_logit", "alpha")


def _case(kind, B, H, T, D, J, io="bf16", temporal=False, gate="none", stats=False, recall=False, name=None):
    c = {"kind": kind, "B": B, "H": H, "T": T, "D": D, "J": J, "io": io, "temporal": temporal, "gate": gate, "stats": stats,
         "recall": recall}
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # one user of the 374M language model (8 heads of 64, four components): a token at a time
        _case("decode", 1, 8, 1, 64, 4, name="decode_one"),
        # a server's batch of that model as the paper trains it, with one decay per key dimension
        _case("decode", 64, 8, 1, 64, 4, gate="key", name="decode_batch"),
        # 256 streams of a model with 32 heads of 128 (the batched-decode configuration): all of the state moves
        _case("decode", 256, 32, 1, 128, 4, name="decode_streams"),
        # short prompts, or the tail of a prompt fed in pieces
        _case("prefill", 2, 8, 37, 64, 4, name="prompt_short"),
        # one user's long prompt: few rows, many tokens
        _case("prefill", 1, 8, 2011, 64, 4, name="prompt_one"),
        # the language-model shaped prefill that the benchmark's headline is quoted on
        _case("prefill", 4, 16, 8192, 128, 4, name="lm_prefill"),
        # a training forward pass of the 374M model's layer, with the sums of the load-balancing loss
        _case("prefill", 16, 8, 2048, 64, 4, stats=True, name="lm_train"),
        # the same kind of layer with the decay per key dimension of the paper's language models (App. D.3)
        _case("prefill", 8, 16, 2048, 64, 4, gate="key", name="lm_gated"),
        # Temporal SwiLA on wide heads, a length that is no multiple of anything
        _case("prefill", 2, 16, 4001, 128, 4, temporal=True, name="lm_temporal"),
        # associative recall in fp32 with eight components (the recall configuration)
        _case("prefill", 64, 4, 512, 64, 8, io="fp32", recall=True, name="recall_fp32"),
        # the layer on raw projections, output norm included
        _case("layer", 4, 8, 3000, 64, 4, name="layer_raw"),
        # host tensors in, host tensors out
        _case("host", 4, 8, 2048, 64, 4, name="host_prefill"),
    ]


def _spread(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("decode", "decode", "prompt", "train", "gated", "fp32", "layer", "host"))
    if kind == "decode":
        H, D = rng.choice(((8, 64), (16, 64), (16, 128), (32, 128)))
        return _case("decode", _spread(rng, 1, 256), H, 1, D, rng.choice((4, 4, 8)) if D == 64 else 4,
                     temporal=rng.random() < 0.25, gate=rng.choice(("none", "none", "key", "out")))
    if kind == "prompt":
        return _case("prefill", rng.choice((1, 1, 2, 3)), rng.choice((8, 16)), _spread(rng, 12, 4096), rng.choice((64, 128)), 4,
                     temporal=rng.random() < 0.25)
    D = rng.choice((64, 64, 128))
    J = rng.choice((4, 4, 8))
    H = rng.choice((4, 8, 16))
    T = _spread(rng, 200, 8192)
    state = J * D * D
    if kind == "train":  # at most half of the language-model shaped prefill's work
        B = _spread(rng, 1, max(1, min(32, int(1.7e10 / (H * T * state)))))
        return _case("prefill", B, H, T, D, J, temporal=rng.random() < 0.25, stats=rng.random() < 0.5)
    B = _spread(rng, 1, max(1, min(64, int(4.3e9 / (H * T * state)))))
    if kind == "gated":
        return _case("prefill", B, H, T, D, J, gate=rng.choice(("key", "key", "out", "component")), temporal=rng.random() < 0.2)
    if kind == "fp32":
        return _case("prefill", B, H, T, D, rng.choice((2, J)), io="fp32", recall=rng.random() < 0.5)
    return _case(kind, B, H, T, D, J)


def _workload(c):
    w = wl.Workload("case", 0, c["B"], c["H"], c["T"], c["D"], c["D"], c["J"], io_dtype=c["io"])
    w = w.variant(temporal=c["temporal"], gated=c["gate"] != "none", granularity=GRANULARITY[c["gate"]])
    return w.with_(flags=w.flags | wl.FLAG_QKV_ACT) if c["kind"] == "layer" else w


def _inputs(c, w, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    B, H, T, D, J, io = w.B, w.H, w.T, w.Dk, w.J, w.torch_io_dtype

    def randn(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    silu = torch.nn.functional.silu
    unit = lambda x: torch.nn.functional.normalize(x, dim=-1)  # noqa: E731
    if c["kind"] == "layer":
        q, k, v = randn(B, H, T, D), randn(B, H, T, D), randn(B, H, T, D)
    elif c["recall"]:  # 64 key-value pairs per sequence, revisited in shuffled order; queries equal keys
        P = min(64, T)
        keys, vals = unit(randn(B, H, P, D)), randn(B, H, P, D)
        at = torch.rand((B, H, -(-T // P), P), generator=g, device="cuda").argsort(dim=-1).reshape(B, H, -1, 1)[:, :, :T]
        k, v = keys.gather(2, at.expand(B, H, T, D)), vals.gather(2, at.expand(B, H, T, D))
        q = k.clone()
    else:
        q, k, v = unit(silu(randn(B, H, T, D))), unit(silu(randn(B, H, T, D))), silu(randn(B, H, T, D))
    inp = {"q": q.to(io), "k": k.to(io), "v": v.to(io), "gk_logit": None, "gq_logit": None, "alpha": None}
    for n in ("beta_logit", "pik_logit", "piq_logit"):
        inp[n] = (0.9 * randn(B, H, T, J, D)).to(io)
    if w.temporal:
        for n in ("gk_logit", "gq_logit"):
            inp[n] = (0.9 * randn(B, H, T, D)).to(io)
    if w.gated:
        shape = (B, H, T, J) if c["gate"] == "component" else (B, H, T, J, D)
        inp["alpha"] = torch.sigmoid(3.0 + randn(*shape))
    return {n: (x if x is None else x.contiguous()) for n, x in inp.items()}


def prepare(case, seed):
    w = _workload(case)
    inp = _inputs(case, w, seed)
    s = {"kind": case["kind"], "w": w, "inp": inp, "stats": None}
    s["o"] = torch.empty((w.B, w.H, w.T, w.Dv), device="cuda", dtype=w.torch_io_dtype)
    s["state"] = binding.state_alloc(w)
    if case["kind"] == "decode":  # a state that a sequence has been written into
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) + 7919)
        s["state"]["W"].normal_(0.0, 0.3, generator=g)
    if case["stats"]:
        s["stats"] = binding.stats_alloc(w)
    if case["kind"] == "layer":
        s["weight"] = 1.0 + 0.1 * torch.randn(w.Dv, device="cuda", generator=torch.Generator(device="cuda").manual_seed(int(seed) + 1))
    if case["kind"] == "host":
        s["inp"] = {n: (x if x is None else x.cpu().pin_memory()) for n, x in inp.items()}
        s["o"] = torch.empty(s["o"].shape, dtype=s["o"].dtype).pin_memory()
        s["state"] = {n: (x if x is None else torch.empty(x.shape, dtype=x.dtype).pin_memory()) for n, x in s["state"].items()}
        s["workspace"] = torch.empty(binding.host_workspace_bytes(w), device="cuda", dtype=torch.uint8)
    return s


def run(state):
    w, inp, o, st = state["w"], state["inp"], state["o"], state["state"]
    kind = state["kind"]
    if kind == "decode":
        binding.swila_decode_step(w, inp, st, o=o)
    elif kind == "host":
        binding.swila_forward_host(w, inp, state["workspace"], state_out=st, o=o)
    elif state["stats"] is not None:
        binding.swila_forward_stats(w, inp, state["stats"], state_out=st, o=o)
    else:
        binding.swila_forward(w, inp, state_out=st, o=o)
        if kind == "layer":
            binding.swila_output_norm(w, o, state["weight"])
    return {"o": o, "state": st, "stats": state["stats"]}


def work(case):
    """Every input once, every output once; three multiply-adds per state element and token (prediction, update, readout),
    and one multiplication more where a decay is applied."""
    w = _workload(case)
    es = 2 if w.io_dtype == "bf16" else 4
    per_token = (2 * w.Dk + 2 * w.Dv + 3 * w.J * w.Dv + (2 * w.Dv if w.temporal else 0)) * es
    per_token += 4 * w.J * {"none": 0, "key": w.Dk, "out": w.Dv, "component": 1}[case["gate"]]
    rows = w.J * w.Dv
    carried = 4 * rows * (w.Dk + (2 if w.temporal else 0))
    heads = w.B * w.H
    moved = heads * (w.T * per_token + carried * (2 if case["kind"] == "decode" else 1))
    if case["stats"]:
        moved += heads * 2 * 4 * 2 * (rows + w.Dv)  # added to: read and written
    if case["kind"] == "layer":
        moved += 4 * w.Dv
    return {"bytes": moved, "flops": heads * w.T * rows * w.Dk * (7.0 if w.gated else 6.0)}


def tolerance(case):
    """bf16 outputs round to 8 bits; fp32 ones carry the rounding of a few hundred dependent updates."""
    return {"rel": 1e-5, "max": 1e-4} if case["io"] == "fp32" else {"rel": 4e-3, "max": 2e-2}
