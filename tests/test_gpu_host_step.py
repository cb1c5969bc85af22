"""Steps on host weights (``ciera_roundtrip_host``): what a copy that the runtime refuses leaves behind, buffers that
overlap, several threads and streams; against the oracle, tolerance 0.

A copy is made to fail on the host: the runtime refuses a range that is page-locked at both ends and not in the middle."""
import ctypes
import mmap

import numpy as np
import pytest
import torch

from harness import OracleTable, compare_caches, compare_recon, compare_step, sender_scratch_is_clean, to_dev_bytes
from paper_2609_04609_b200 import workloads as wl

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SIZES = [8192 * 40 + 3, 100, 8192 * 900 + 4097, 8192 * 12 + 5, 1_000_000]  # about 18 MB in bf16: four parts


class HalfPinned:
    """Host memory of ``size`` bytes of which only the first and the last quarter are page-locked."""

    def __init__(self, size):
        page = mmap.PAGESIZE
        self.map = mmap.mmap(-1, (size + page - 1) // page * page)
        self.tensor = torch.frombuffer(self.map, dtype=torch.uint8)[:size]
        base, quarter = self.tensor.data_ptr(), len(self.map) // 4 // page * page
        self.locked = [(base, quarter), (base + len(self.map) - quarter, quarter)]
        for at, n in self.locked:
            assert int(torch.cuda.cudart().cudaHostRegister(at, n, 0)) == 0

    def release(self):
        for at, _ in self.locked:
            assert int(torch.cuda.cudart().cudaHostUnregister(at)) == 0


def _make(sizes=SIZES, block=512, seed=3, steps=3):
    from paper_2609_04609_b200 import runtime

    codec = runtime.LayerCodec.from_tensors(sizes, 1, "bf16", block, DEV)
    table = OracleTable(codec.units, 0, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(seed)
    w = [wl.init_weights(codec.weights_bytes // 2, "bf16", gen)]
    for _ in range(steps):
        w.append(wl.step_clustered(w[-1], gen, f=0.3))
    bits = [wl.as_bits(x) for x in w]
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    staging = torch.empty(codec.weights_bytes, dtype=torch.uint8, device=DEV)
    return codec, table, bits, staging


def _pinned(bits):
    return torch.from_numpy(bits.view(np.uint8).copy()).pin_memory()


def _compare(codec, table, exp, bits, label):
    torch.cuda.synchronize()
    codec.check_status()
    compare_step(codec, exp, bits, label)
    compare_caches(codec, table, label)
    compare_recon(codec, exp, bits, 0, label)


@pytest.mark.parametrize("side", ["in", "out"])
def test_a_copy_that_fails_half_way(side):
    from paper_2609_04609_b200 import ciera

    codec, table, bits, staging = _make()
    good_out = torch.zeros(codec.weights_bytes, dtype=torch.uint8).pin_memory()
    holed = HalfPinned(codec.weights_bytes)
    holed.tensor.copy_(torch.from_numpy(bits[1].view(np.uint8)))
    before = codec.sender_cache.clone(), codec.receiver_cache.clone()
    with pytest.raises(ciera.CieraError) as e:
        if side == "in":
            codec.step_host(holed.tensor, good_out, staging)
        else:
            codec.step_host(_pinned(bits[1]), holed.tensor, staging)
    assert e.value.status == ciera.ERR_CUDA
    torch.cuda.synchronize()
    holed.release()
    assert sender_scratch_is_clean(codec)
    if side == "in":  # nothing was stepped
        assert torch.equal(codec.sender_cache, before[0]) and torch.equal(codec.receiver_cache, before[1])
    else:  # the step on the device is complete
        _compare(codec, table, table.step(bits[1]), bits[1], "step whose way out failed")
    for t in (2, 3):
        codec.step_host(_pinned(bits[t]), good_out, staging)
        _compare(codec, table, table.step(bits[t]), bits[t], f"t={t}")
    ciera.cache_init(codec.plan, codec.sender_cache, staging)  # (the earlier error is not reported twice)


@pytest.mark.parametrize("shift", [-(1 << 20), 0, 16, 1 << 20, 8 << 20])
def test_host_ranges_that_overlap(shift):
    """The step reads all of its weights before it writes any: the output may lie over the input, shifted or not."""
    codec, table, bits, staging = _make(steps=1)
    n = codec.weights_bytes
    room = torch.zeros(n + (9 << 20), dtype=torch.uint8).pin_memory()
    src, out = room[1 << 20 :][:n], room[(1 << 20) + shift :][:n]
    src.copy_(torch.from_numpy(bits[1].view(np.uint8)))
    codec.step_host(src, out, staging)
    _compare(codec, table, table.step(bits[1]), bits[1], f"shift {shift}")
    for u in codec.units:
        lo, hi = int(u["weights_off"]), int(u["weights_off"]) + 2 * int(u["n_values"])
        assert np.array_equal(out.numpy()[lo:hi], bits[1].view(np.uint8)[lo:hi])


def test_two_threads_on_one_plan():
    """Steps in parts from two threads on one plan, each with a stream and buffers of its own, at the same time."""
    import threading

    from paper_2609_04609_b200 import ciera, runtime

    first, table0, bits0, staging0 = _make(seed=5, steps=4)
    second, table1, bits1, staging1 = _make(seed=6, steps=4)
    second.plan = first.plan  # (the same table of units)
    jobs = [(first, table0, bits0, staging0), (second, table1, bits1, staging1)]
    errors = []

    def work(codec, table, bits, staging):
        try:
            stream = torch.cuda.Stream()
            out = torch.zeros(codec.weights_bytes, dtype=torch.uint8).pin_memory()
            for t in range(1, len(bits)):
                src = _pinned(bits[t])
                exp = table.step(bits[t])
                codec.step_host(src, out, staging, stream=stream)
                stream.synchronize()
                codec.check_status()
                compare_step(codec, exp, bits[t], f"t={t}")
                compare_recon(codec, exp, bits[t], 0, f"t={t}")
                for u in codec.units:
                    lo, hi = int(u["weights_off"]), int(u["weights_off"]) + 2 * int(u["n_values"])
                    assert np.array_equal(out.numpy()[lo:hi], bits[t].view(np.uint8)[lo:hi]), f"t={t}"
        except Exception as e:  # (reported by the main thread)
            errors.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    assert not errors, errors
    for codec, table, bits, _ in jobs:
        compare_caches(codec, table, "threads")


def test_more_streams_than_the_library_keeps_copy_streams_for():
    """Twelve codecs, a stream each, stepped round and round without waiting in between; plans come and go meanwhile."""
    from paper_2609_04609_b200 import runtime

    made = [_make([8192 * 300 + i, 4099], seed=20 + i, steps=2) for i in range(12)]
    streams = [torch.cuda.Stream() for _ in made]
    outs = [torch.zeros(m[0].weights_bytes, dtype=torch.uint8).pin_memory() for m in made]
    srcs = [[_pinned(b) for b in m[2]] for m in made]
    torch.cuda.synchronize()
    for t in (1, 2, 1, 2):
        for i, (codec, _, _, staging) in enumerate(made):
            codec.step_host(srcs[i][t], outs[i], staging, stream=streams[i])
    torch.cuda.synchronize()
    for i, (codec, table, bits, _) in enumerate(made):
        codec.check_status()
        for t in (1, 2, 1, 2):
            exp = table.step(bits[t])
        compare_step(codec, exp, bits[2], f"codec {i}")
        compare_caches(codec, table, f"codec {i}")
        compare_recon(codec, exp, bits[2], 0, f"codec {i}")
    del made, codec, table
    codec, table, bits, staging = _make(steps=1)  # after the last plan went, and its streams with it
    out = torch.zeros(codec.weights_bytes, dtype=torch.uint8).pin_memory()
    codec.step_host(_pinned(bits[1]), out, staging)
    _compare(codec, table, table.step(bits[1]), bits[1], "fresh")
