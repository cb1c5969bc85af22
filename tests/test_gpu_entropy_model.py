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


@pytest.mark.parametrize("dtype", [0, 2])
@pytest.mark.parametrize("n_units,size", [(148, 4096), (149, 4096), (741, 4096), (149, 65_500), (297, 65_500), (296, 4096), (296, 65_500),
                                          (740, 4096), (160, 131_072)])
def test_numbers_of_units(n_units, size, dtype):
    """A thread block of 32 warps per unit up to one per SM, of 16 up to two, narrow ones beyond, and those in two builds
    by their number."""
    from paper_2609_04609_b200 import runtime

    name = {0: "bf16", 2: "fp16"}[dtype]
    codec = guard(runtime.LayerCodec.from_tensors([size + 37 * (i % 5) for i in range(n_units)], 1, name, 64, DEV, slack=256))
    gen = torch.Generator().manual_seed(n_units)
    w = (torch.randn(codec.weights_bytes // 2, generator=gen) * 0.02).to({0: torch.bfloat16, 2: torch.float16}[dtype])
    bits = w.view(torch.int16).numpy().view(np.uint16)
    codec.init_caches(None)
    codec.encode(to_dev_bytes(bits, DEV))
    codec.entropy_encode()
    torch.cuda.synchronize()
    sent, wire = codec.msg_send.cpu().numpy(), codec.wire_bytes.cpu().numpy().copy()
    codec.transport()
    codec.entropy_decode()
    torch.cuda.synchronize()
    codec.check_status()
    back, raw_wire = codec.msg_recv.cpu().numpy(), codec.wire_bytes.cpu().numpy()
    for i, u in enumerate(codec.units):
        n, lo, mo = int(u["n_values"]), int(u["weights_off"]) // 2, int(u["msg_off"])
        raw = ora.encode(bits[lo : lo + n], np.zeros(n, np.uint8), dtype, 64)[0]
        want = rans.entropy_encode_message(raw, n, dtype, 64)
        assert want.size < raw.size and int(wire[i]) == want.size and int(raw_wire[i]) == raw.size
        assert np.array_equal(sent[mo : mo + want.size], want) and np.array_equal(back[mo : mo + raw.size], raw)
    codec.canaries.check("units")


@pytest.mark.parametrize("chunks", [92, 100, 200, 400])
def test_chunks_of_long_units_in_parts(chunks):
    """One long unit of so many chunks that each is the work of 8, 8, 4 and 2 thread blocks: coded shorter, restored."""
    from paper_2609_04609_b200 import runtime

    codec = runtime.LayerCodec.from_tensors([262_144 * (chunks - 1) + 4097], 1, "bf16", 512, DEV)
    gen = torch.Generator(DEV).manual_seed(chunks)
    w = (torch.randn(codec.weights_bytes // 2, generator=gen, device=DEV) * 0.02).bfloat16().view(torch.uint8)
    codec.init_caches(None)
    codec.encode(w)
    raw_wire = int(codec.wire_bytes[0])
    raw = codec.msg_send[:raw_wire].clone()
    codec.entropy_encode()
    coded = int(codec.wire_bytes[0])
    assert coded < 0.75 * raw_wire
    codec.transport()
    codec.entropy_decode()
    codec.decode()
    torch.cuda.synchronize()
    codec.check_status()
    assert int(codec.wire_bytes[0]) == raw_wire and torch.equal(codec.msg_recv[:raw_wire], raw)
    n = 2 * int(codec.units[0]["n_values"])
    assert torch.equal(codec.weights_out[:n], w[:n])
