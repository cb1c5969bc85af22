"""The work that a program using this codec has it do, as a list of cases with sizes.

A case is a table of tensors, cut into shards, and what is done with it in one training iteration:

* ``step``      ``LayerCodec.step``: sender, transport stand-in and receiver of one table
* ``pipeline``  ``LayerPipeline.step``: the same over a stack of tables on two streams
* ``sender``    ``LayerCodec.encode``: one rank's sending side alone
* ``receiver``  ``LayerCodec.decode``: the receiving side alone, on messages that have arrived
* ``hashed``    ``LayerCodec.encode_hashed``: the sending side that keeps a hash per block
* ``entropy``   a step with the entropy stage before and after the transport
* ``host``      ``LayerCodec.step_host``: a whole step on weights that live in pinned host memory

Two consecutive iterates A and B of a synthetic weight trajectory stay on the device; a pass works on
the one that the caches do not hold, so every pass is a real step (the set of changed exponents is the
same in both directions).  Everything is integer and bit work: results are exact.
"""
from __future__ import annotations

from typing import List

import torch

from paper_2609_04609_b200 import ciera, runtime
from paper_2609_04609_b200 import workloads as wl

DEVICE = "cuda:0"
ADAM_RATE = 0.034  # share of the exponents that one Adam-like step changes on N(0, 0.02) weights
GAUSSIAN_RATE = 0.027
EXPERT = "3*2097152"  # gate, up and down of one OLMoE-shaped expert (2048 x 1024 each)
LAYER = "192*2097152"  # 64 experts: one OLMoE-shaped MoE layer
DENSE = ",".join(str(n) for n in wl.dense_tensor_sizes())  # dense tensors of 4 KB ... 256 MB in bf16


def _case(name, kind, tensors, shards, dtype, block, update, rate=0.0, segment=0, layers=1):
    return {"name": name, "kind": kind, "tensors": tensors, "shards": shards, "dtype": dtype, "block": block,
            "update": update, "rate": rate, "segment": segment, "layers": layers}


def listed():
    return [
        # the smallest table anybody steps: one 1024 x 512 matrix on 4 shards; launches and latency count
        _case("matrix_step_bf16", "step", "524288", 4, "bf16", 512, "gaussian"),
        # a handful of tensors of odd sizes: shards end inside tiles and blocks, some are long
        _case("ragged_step_bf16", "step", "3000005,131072,70001", 2, "bf16", 512, "adam"),
        # one expert on 16 shards: what a rank steps when experts are gathered one at a time
        _case("expert_step_bf16", "step", EXPERT, 16, "bf16", 512, "clustered", 0.22),
        # one whole MoE layer, the unit of work of a layer-wise gather, at the paper's block change rate
        _case("layer_step_bf16", "step", LAYER, 16, "bf16", 512, "clustered", 0.22),
        # several layers in a row, the sender of one beside the receiver of the one before
        _case("stack_pipeline_bf16", "pipeline", LAYER, 16, "bf16", 512, "clustered", 0.22, layers=4),
        # master weights kept in fp32
        _case("layer_step_fp32", "step", LAYER, 16, "fp32", 512, "clustered", 0.22),
        # fine-grained experts and dense tensors of all sizes in one table; changes spread over all values
        _case("mixed_step_bf16", "step", "768*1048576," + DENSE, 8, "bf16", 512, "inject", 0.01),
        # change detection per value: the setting that compresses when every value moves on its own
        _case("values_step_bf16", "step", LAYER, 16, "bf16", 1, "adam"),
        # fp16 weights, the receiving side alone, at the paper's smallest block size
        _case("layer_receiver_fp16", "receiver", LAYER, 16, "fp16", 64, "clustered", 0.22),
        # the paper's own sender: a 128-bit hash per block in place of the previous exponents
        _case("layer_hashed_bf16", "hashed", LAYER, 16, "bf16", 512, "clustered", 0.22),
        # slow links: the changed exponents are entropy-coded as well
        _case("layer_entropy_bf16", "entropy", LAYER, 16, "bf16", 512, "clustered", 0.22),
        # eight experts whose weights live in pinned host memory (an offloaded optimizer)
        _case("experts_host_bf16", "host", "24*2097152", 16, "bf16", 512, "clustered", 0.22),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "pipeline", "sender", "receiver", "hashed", "entropy", "host"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "fp32", "fp16"])
    coarse = kind in ("hashed", "pipeline", "host")
    block = 1 << (rng.randint(5, 12) if coarse or rng.random() < 0.75 else rng.randint(0, 4))
    layers = rng.randint(2, 4) if kind == "pipeline" else 1
    # 2^17 ... 2^28 values in all (host memory: 2^25), in 1 ... 192 tensors of at least 2^11 values
    total = 2.0 ** rng.uniform(17, 25 if kind == "host" else 28) / layers
    count = int(min(2.0 ** rng.uniform(0, 7.6), total / 2048)) or 1
    numel = max(2048, int(total / count))
    if rng.random() < 0.5:  # matrices of whole rows
        numel = max(2048, numel // 1024 * 1024)
    tensors = "%d*%d" % (count, numel)
    if rng.random() < 0.5:  # and a small tensor of odd size
        tensors += ",%d" % rng.randint(1001, 100_001)
    shards = rng.choice([1, 2, 4, 8, 16, 32, 64])
    update = rng.choice(["clustered", "clustered", "adam", "inject"])
    rate = {"clustered": rng.uniform(0.05, 0.5), "adam": 0.0, "inject": 10 ** rng.uniform(-3, -0.3)}[update]
    segment = 512 if update == "inject" and rng.random() < 0.5 else 0
    return {"kind": kind, "tensors": tensors, "shards": shards, "dtype": dtype, "block": block, "update": update,
            "rate": round(rate, 4), "segment": segment, "layers": layers}


def numels(case) -> List[int]:
    out: List[int] = []
    for part in case["tensors"].split(","):
        count, _, numel = part.rpartition("*")
        out += [int(numel)] * int(count or 1)
    return out


def _next(case, w, gen):
    if case["update"] == "gaussian":
        return wl.step_gaussian(w, gen)
    if case["update"] == "adam":
        return wl.step_adam_like(w, gen)
    if case["update"] == "clustered":
        return wl.step_clustered(w, gen, f=case["rate"])
    return wl.inject_exponent_changes(w, gen, case["rate"], case["segment"])


def prepare(case, seed):
    state = {"kind": case["kind"], "codecs": [], "iterates": [[], []], "turn": 0}
    for layer in range(case["layers"]):
        codec = runtime.LayerCodec.from_tensors(numels(case), case["shards"], case["dtype"], case["block"], DEVICE)
        gen = wl.make_generator(seed * 1009 + layer, DEVICE)
        a = wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[case["dtype"]], case["dtype"], gen)
        b = _next(case, a, gen)
        a, b = a.view(torch.uint8), b.view(torch.uint8)
        codec.init_caches(a)
        if case["kind"] == "hashed":
            codec.init_hash_cache(a)
        state["codecs"].append(codec)
        state["iterates"][0].append(b)  # the caches hold A: the first pass works on B
        state["iterates"][1].append(a)
    if case["kind"] == "pipeline":
        state["pipeline"] = runtime.LayerPipeline(state["codecs"])
    elif case["kind"] == "receiver":
        codec.encode(state["iterates"][0][0])
        codec.transport()
    elif case["kind"] == "host":
        state["host"] = [x[0].cpu().pin_memory() for x in state["iterates"]]
        state["host_out"] = torch.zeros_like(state["host"][0]).pin_memory()
        state["staging"] = torch.empty_like(a)
    return state


def run(state):
    codecs, kind = state["codecs"], state["kind"]
    weights = state["iterates"][state["turn"]]
    codec, w = codecs[0], weights[0]
    if kind == "step":
        codec.step(w)
    elif kind == "pipeline":
        state["pipeline"].step(weights)
        state["pipeline"].wait()
    elif kind == "sender":
        codec.encode(w)
    elif kind == "receiver":
        codec.decode()
    elif kind == "hashed":
        codec.encode_hashed(w)
    elif kind == "entropy":
        codec.encode(w)
        codec.entropy_encode()
        codec.transport()
        codec.entropy_decode()
        codec.decode()
    else:
        codec.step_host(state["host"][state["turn"]], state["host_out"], state["staging"])
    state["turn"] ^= 1
    out = []
    for c in codecs:
        got = {"wire_bytes": c.wire_bytes, "changed_blocks": c.changed_blocks}
        if kind in ("sender", "hashed"):
            got["messages"] = c.msg_send
        else:
            got.update(messages=c.msg_recv, weights=c.weights_out, receiver_cache=c.receiver_cache)
        if kind == "hashed":
            got["hash_cache"] = c.hash_cache
        elif kind != "receiver":
            got["sender_cache"] = c.sender_cache
        if kind == "host":
            got["weights"] = state["host_out"]
        out.append(got)
    return out


def _changed_share(case) -> float:
    """Expected share of the exponents that travel (those of changed blocks)."""
    block, rate = case["block"], case["rate"]
    if case["update"] == "gaussian":
        return 1 - (1 - GAUSSIAN_RATE) ** block
    if case["update"] == "adam":
        return 1 - (1 - ADAM_RATE) ** block
    if case["update"] == "clustered":
        hit = 1 - (1 - ADAM_RATE) ** min(block, 512)
        return 1 - (1 - rate * hit) ** max(1, block // 512)
    if case["segment"]:
        return 1 - (1 - rate) ** max(1, block // case["segment"])
    return 1 - (1 - rate) ** block


def work(case):
    n = case["layers"] * sum(numels(case))
    block, q, kind = case["block"], _changed_share(case), case["kind"]
    value, sm, ex = {"bf16": (2, 1, 1), "fp32": (4, 3, 1), "fp16": (2, 11 / 8, 5 / 8)}[case["dtype"]]
    message = sm + 1 / (8 * block) + q * ex  # bytes per value on the wire
    # sender: weights and cached exponents in, message and refreshed exponents out
    sender = value + 1 + message + q
    if kind == "hashed":
        sender = value + message + 16 * (1 + q) / block
    # receiver: message and the unchanged blocks' cached exponents in, weights and refreshed exponents out
    receiver = message + (1 - q) + value + q
    # a whole step writes the message on both sides, but need not fetch what it has just written
    total = {"sender": sender, "hashed": sender, "receiver": receiver}.get(kind, sender + receiver)
    if kind == "host":
        total += 2 * value  # over the link, in and out
    return {"bytes": n * total, "flops": 0}


def tolerance(case):
    return "exact"
