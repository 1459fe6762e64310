"""What a user of this framework has it do: one MoE layer on one GPU, from a single token to a long prefill.

A case names the layer's shape, the number of tokens, the skew of the router and the entry point:

  forward   WeaveMoE.forward(x, logits) on a handle that the program keeps, inputs and output on the GPU
  static    forward_static(), no handle and no workspace, into a buffer that the caller owns
  ep        forward() of a handle that acts as one rank of an expert-parallel group of `ranks`
  host      forward_host_pipelined() over `batches` batches in pinned host memory, then host_wait()

The shapes are those of this repository's workloads (workloads/__init__.py) and the inputs follow its recipe:
x ~ N(0,1) in bf16, weights ~ N(0,0.02) in bf16, router logits ~ N(0,1) in fp32, with a bias of
-s * ln(rank + 1) for a Zipf-like load of the experts where the case has a skew s > 0.
"""
import math

import numpy as np
import torch

import paper_2609_21483_b200 as weave

# name -> hidden, expert FFN width, routed experts, experts per token, shared experts
SHAPES = {
    "tiny": (512, 1024, 8, 2, 0),
    "mixtral": (4096, 14336, 8, 2, 0),
    "qwen3_30b": (2048, 768, 128, 8, 0),
    "dsv2lite": (2048, 1408, 64, 6, 2),
    "qwen3_235b": (4096, 1536, 128, 8, 0),
    "phi35": (4096, 6400, 16, 2, 0),
    "qwen35_35b": (2048, 512, 256, 8, 0),
    "dsv2": (5120, 1536, 160, 6, 0),
    "dsv3": (7168, 2048, 256, 8, 0),
}
MAX_T = 16384            # the longest batch of the repository's workloads
MAX_T_STATIC = 256       # ... and of its runs through forward_static (the built-in scratch is 64 MiB)
SKEWS = (0.0, 0.5, 0.8, 1.2, 1.6)


def _case(name, shape, T, skew=0.0, entry="forward", ranks=1, rank=0, batches=1):
    return {"name": name, "shape": shape, "T": T, "skew": skew, "entry": entry, "ranks": ranks, "rank": rank,
            "batches": batches}


def listed():
    return [
        # decode: one sequence, a few, a few dozen, with the routers of many small experts
        _case("decode_1", "qwen3_30b", 1),
        _case("decode_7", "dsv2lite", 7),
        _case("decode_27", "qwen3_30b", 27, 0.5),
        # decode-like batches of the shape with shared experts
        _case("decode_64", "dsv2lite", 64),
        _case("decode_256", "dsv2lite", 256),
        # the smallest layer, for callers that may not allocate
        _case("tiny_static", "tiny", 256, entry="static"),
        # a ragged prefill chunk over many small experts
        _case("chunk_1023", "qwen35_35b", 1023, 0.5),
        # batches that live in host memory, streamed through the layer
        _case("host_4x512", "dsv2lite", 512, entry="host", batches=4),
        # prefill: few large experts; many small ones with a skewed load; the largest layer
        _case("prefill_mixtral", "mixtral", 4096),
        _case("prefill_skewed", "qwen3_30b", 8192, 1.2),
        _case("prefill_235b", "qwen3_235b", 16384, 1.2),
        # one rank's share of that layer in a group of four
        _case("ep_share", "qwen3_235b", 16384, 1.2, entry="ep", ranks=4, rank=1),
    ]


def draw(rng):
    largest = work(listed()[-2])
    while True:
        shape = rng.choice(sorted(SHAPES))
        H, I, E, k, S = SHAPES[shape]
        entry = rng.choice(("forward", "forward", "forward", "forward", "static", "ep", "host"))
        top = MAX_T_STATIC if entry == "static" else MAX_T
        T = min(top, int(round(math.exp(rng.uniform(0.0, math.log(top))))))
        c = {"shape": shape, "T": T, "skew": rng.choice(SKEWS), "entry": entry, "ranks": 1, "rank": 0, "batches": 1}
        if entry == "static" and weave.workspace_bytes(H, I, E, k, S, T) > weave.load().weave_moe_static_scratch_bytes():
            continue
        if entry == "ep":
            ranks = rng.choice((2, 4, 8))
            if S or E // ranks < k or T < 64:
                continue
            c["ranks"], c["rank"] = ranks, rng.randrange(ranks)
        if entry == "host":
            c["batches"] = rng.choice((1, 2, 4))
            if T * c["batches"] > MAX_T:
                continue
        w = work(c)
        if w["bytes"] <= largest["bytes"] and w["flops"] <= largest["flops"]:
            return c


def _normal(shape, gen, std, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)


def prepare(case, seed):
    H, I, E, k, S = SHAPES[case["shape"]]
    T, entry = case["T"], case["entry"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    gate_up = _normal((E + S, 2 * I, H), gen, 0.02, torch.bfloat16)
    down = _normal((E + S, H, I), gen, 0.02, torch.bfloat16)
    n = T * case["batches"]
    x = _normal((n, H), gen, 1.0, torch.bfloat16)
    logits = _normal((n, E), gen, 1.0, torch.float32)
    if case["skew"] > 0:
        rank = torch.randperm(E, generator=gen, device="cuda").float()
        logits -= case["skew"] * torch.log(rank + 1.0)
    state = {"entry": entry, "x": x, "logits": logits, "gate_up": gate_up, "down": down, "E": E, "k": k, "S": S}
    if entry == "static":
        state["out"] = torch.empty_like(x)
        return state
    moe = weave.WeaveMoE(gate_up, down, E, k, S, max_tokens=T)
    if entry == "ep":
        moe.set_expert_parallel(case["rank"], case["ranks"])
    if entry == "host":
        # the batches are host data: the device copies they were made from are not part of the state
        del state["x"], state["logits"]
        state["x_host"] = [b.cpu().pin_memory() for b in x.split(T)]
        state["logits_host"] = [b.cpu().pin_memory() for b in logits.split(T)]
        state["out_host"] = [torch.empty_like(b).pin_memory() for b in state["x_host"]]
    state["moe"] = moe
    return state


def run(state):
    if state["entry"] == "static":
        return weave.forward_static(state["x"], state["logits"], state["gate_up"], state["down"], state["E"], state["k"],
                                    state["S"], out=state["out"])
    moe = state["moe"]
    if state["entry"] == "host":
        for x, logits, out in zip(state["x_host"], state["logits_host"], state["out_host"]):
            moe.forward_host_pipelined(x, logits, out)
        moe.host_wait()
        return state["out_host"]
    return moe.forward(state["x"], state["logits"])


def _routed(case):
    """(token, expert) pairs and experts with at least one of them, for one batch of inputs like prepare()'s."""
    H, I, E, k, S = SHAPES[case["shape"]]
    T = case["T"]
    rng = np.random.default_rng(12345)
    logits = rng.standard_normal((T, E), dtype=np.float32)
    logits -= np.float32(case["skew"]) * np.log(np.arange(1, E + 1, dtype=np.float32))
    idx = np.argpartition(-logits, k - 1, axis=1)[:, :k].ravel()
    if case["ranks"] > 1:
        # which rank holds the busy experts is the permutation's choice: count an average rank's share
        counts = np.bincount(rng.permutation(E)[idx], minlength=E).reshape(case["ranks"], -1)
        return float(counts.sum()) / case["ranks"], float((counts > 0).sum()) / case["ranks"]
    return float(idx.size), float(np.unique(idx).size)


def work(case):
    """The layer as one function: the selected experts' weights, x, the logits and the output once, and three
    H x I products for each (token, expert) pair.  The host entry point reads the weights once per batch."""
    H, I, E, k, S = SHAPES[case["shape"]]
    T, b = case["T"], case["batches"]
    pairs, experts = _routed(case)
    pairs, experts = pairs + T * S, experts + S
    return {"bytes": b * (experts * 3.0 * H * I * 2 + 2.0 * T * H * 2 + 4.0 * T * E), "flops": b * pairs * 6.0 * H * I}


def tolerance(case):
    """Three roundings to bf16 lie between the inputs and the result (the gated product, each expert's output, the
    sum).  Against the layer in 64 bits the relative error is 2.8e-3 to 2.9e-3 over the cases up to 1023 tokens, and
    the largest difference 0.9e-2 to 1.5e-2 of the result's root mean square or of the value; about four times that
    is allowed."""
    return {"rel": 1.2e-2, "max": 6e-2}
