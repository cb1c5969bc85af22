"""The entropy coder's arithmetic at the edges of its model: every kind of reciprocal (frequency 1, powers of two, the
round-up and the round-down kind, 4096 alone), tables in which one symbol owns nearly all slots, and payload lengths
around the groups of 128 and 512 symbols the coder takes at once and around the segment of 4096.  Coded bytes and
lengths against the oracle, then the raw payload restored: tolerance 0."""
import numpy as np
import pytest
import torch

from harness import guard, to_dev_bytes
from oracle import ciera_oracle as ora
from oracle import rans_oracle as rans

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _weights(symbols):
    """bf16 bit patterns with the given exponents."""
    return (symbols.astype(np.uint16) << 7) | 5


def _draw(rng, n, freqs):
    s = np.repeat(np.arange(1, len(freqs) + 1), freqs)
    return rng.choice(s, n) if n != 4096 else rng.permutation(np.resize(s, n))


MODELS = [[4096], [4095, 1], [2048, 2048], [2049, 2047], [2731, 1365], [3277, 819], [3001, 1000, 95], [4000] + [1] * 96,
          [2994, 1102], [3024, 1000, 72], [2047, 1025, 1024], [16] * 254 + [32], [1024, 1023, 1, 2048], [2500, 1500, 96], [3500, 500, 96]]


def test_models_and_lengths():
    from paper_2609_04609_b200 import runtime

    rng = np.random.default_rng(9)
    lengths = [4096] * len(MODELS) + [127, 128, 129, 511, 512, 513, 640, 4095, 4097, 4608, 8191, 12288 + 31, 262_144 + 700]
    models = MODELS + [MODELS[i % len(MODELS)] for i in range(len(lengths) - len(MODELS))]
    codec = guard(runtime.LayerCodec.from_tensors(lengths, 1, "bf16", 1, DEV, slack=256))
    w = np.zeros(codec.weights_bytes // 2, np.uint16)
    parts = [_weights(_draw(rng, n, m)) for n, m in zip(lengths, models)]
    for u, part in zip(codec.units, parts):
        lo = int(u["weights_off"]) // 2
        w[lo : lo + part.size] = part
    codec.init_caches(None)  # zero caches: every value's exponent travels
    codec.encode(to_dev_bytes(w, DEV))
    raw = codec.msg_send.cpu().numpy()
    raw_wire = codec.wire_bytes.cpu().numpy().copy()
    codec.entropy_encode()
    torch.cuda.synchronize()
    coded, wire = codec.msg_send.cpu().numpy(), codec.wire_bytes.cpu().numpy()
    kinds = set()
    for i, (u, part) in enumerate(zip(codec.units, parts)):
        mo, n = int(u["msg_off"]), part.size
        po = int(raw_wire[i]) - n
        payload = raw[mo + po : mo + po + n]
        assert np.array_equal(payload, (part >> 7).astype(np.uint8))
        want = rans.encode(payload)
        if want is None or len(want) >= n:
            want = payload
        assert int(wire[i]) == po + len(want), f"unit {i}: coded length"
        assert np.array_equal(coded[mo + po : mo + po + len(want)], want), f"unit {i}: coded bytes"
        kinds.add(len(want) < n)
    assert kinds == {True, False}
    codec.transport()
    codec.entropy_decode()
    codec.decode()
    torch.cuda.synchronize()
    codec.check_status()
    codec.canaries.check("restored")
    assert np.array_equal(codec.wire_bytes.cpu().numpy(), raw_wire)
    out = codec.weights_out.cpu().numpy().view(np.uint16)
    for u, part in zip(codec.units, parts):
        lo = int(u["weights_off"]) // 2
        assert np.array_equal(out[lo : lo + part.size], part)
