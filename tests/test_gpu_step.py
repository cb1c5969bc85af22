"""The whole step in one launch (``ciera_step``) against the three calls it stands for, and those three against the
oracle: tolerance 0.  Units end at the edges of pieces, warps, blocks and tiles; one is long enough for the look-back
between thread blocks; the block changes from hardly any to every block, so that the receiver's cached exponents come
both staged and straight from memory.  In a second pass the receiver's cache holds other exponents than the sender's:
what comes out then shows that the receiver's part uses its own cache and not the sender's weights."""
import os
import re

import numpy as np
import pytest
import torch

from harness import OracleTable, compare_caches, compare_recon, compare_step, guard, one_launch, three_calls, to_dev_bytes
from paper_2609_04609_b200 import workloads as wl

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
NAME = {0: "bf16", 1: "fp32", 2: "fp16"}
SIZES = [1, 7, 8, 9, 255, 256, 257, 0, 511, 513, 4096, 8191, 8192, 8193, 8192 * 5, 8192 * 12 + 4097, 8192 * 40 + 3]
STATE = ("sender_cache", "receiver_cache", "weights_out", "wire_bytes", "changed_blocks")


@pytest.mark.parametrize("block", [1, 2, 4, 8, 16, 32, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_one_launch_equalsthree_calls_equals_the_oracle(dtype, block):
    from paper_2609_04609_b200 import ciera, runtime

    one, three = (guard(runtime.LayerCodec.from_tensors(SIZES, 1, NAME[dtype], block, DEV, slack=256)) for _ in range(2))
    table = OracleTable(one.units, dtype, block, one.cache_bytes, one.msg_bytes)
    gen = wl.make_generator(31 * block + dtype)
    w = [wl.init_weights(one.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    for model, kw in (("clustered", {"f": 0.1}), ("inject", {"c": 0.9}), ("inject", {"c": 0.0})):
        step = wl.step_clustered if model == "clustered" else wl.inject_exponent_changes
        w.append(step(w[-1], gen, **kw))
    bits = [wl.as_bits(x) for x in w]
    dev = [to_dev_bytes(b, DEV) for b in bits]
    table.init_caches(bits[0])
    for codec in (one, three):
        codec.init_caches(dev[0])
    for t in (1, 2, 3):
        exp = table.step(bits[t])
        launches0 = ciera.kernel_launch_count()
        one.step(dev[t])
        assert ciera.kernel_launch_count() - launches0 == 1
        three_calls(three, dev[t])
        torch.cuda.synchronize()
        for codec in (one, three):
            codec.check_status()
            compare_step(codec, exp, bits[t], f"t={t}")
            compare_caches(codec, table, f"t={t}")
            compare_recon(codec, exp, bits[t], dtype, f"t={t}")
    # the receiver's cache out of step with the sender's
    other = to_dev_bytes(wl.as_bits(wl.init_weights(w[0].numel(), NAME[dtype], gen)), DEV)
    for codec in (one, three):
        ciera.cache_init(codec.plan, codec.receiver_cache, other)
    one.step(dev[1])
    three_calls(three, dev[1])
    torch.cuda.synchronize()
    for codec in (one, three):
        codec.check_status()
        codec.canaries.check("receiver out of step")
    for name in STATE:
        assert torch.equal(getattr(one, name), getattr(three, name)), name
    assert not torch.equal(one.weights_out[: dev[1].numel()], dev[1])
    for u, n in zip(one.units, one.wire_bytes.tolist()):
        lo = int(u["msg_off"])
        for name in ("msg_send", "msg_recv"):
            assert torch.equal(getattr(one, name)[lo : lo + n], three.msg_send[lo : lo + n]), name


def test_in_place():
    """Reconstructed weights may overwrite the weights."""
    from paper_2609_04609_b200 import runtime

    codec = runtime.LayerCodec.from_tensors(SIZES, 2, "bf16", 512, DEV)
    gen = wl.make_generator(5)
    w0 = wl.init_weights(codec.weights_bytes // 2, "bf16", gen)
    w1 = wl.step_clustered(w0, gen, f=0.3)
    codec.init_caches(to_dev_bytes(wl.as_bits(w0), DEV))
    buf = to_dev_bytes(wl.as_bits(w1), DEV)
    want = buf.clone()
    codec.step(buf, buf)
    torch.cuda.synchronize()
    codec.check_status()
    assert torch.equal(buf, want)


@pytest.mark.parametrize("block", [1, 8, 64, 512, 2048, 4096])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_runs_of_short_units(dtype, block):
    """Enough units of five tiles (a run of four, then a run of one) that they are handed out in runs rather than
    spread tile by tile; the three calls, then the whole step, against the oracle."""
    from paper_2609_04609_b200 import runtime

    sizes = [8192 * 5, 8192 * 4 + 1, 8192 * 5 - 1, 8192 * 4 + 4100] * 55 + [100, 8192 * 33 + 5]
    codec = guard(runtime.LayerCodec.from_tensors(sizes, 1, NAME[dtype], block, DEV, slack=256))
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(7 * block + dtype, DEV)
    w = [wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    w += [wl.step_clustered(w[0], gen, f=0.3)]
    bits = [wl.as_bits(x) for x in w]
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    for t, step in ((1, three_calls), (0, one_launch)):
        exp = table.step(bits[t])
        step(codec, to_dev_bytes(bits[t], DEV))
        torch.cuda.synchronize()
        codec.check_status()
        compare_step(codec, exp, bits[t], f"t={t}")
        compare_caches(codec, table, f"t={t}")
        compare_recon(codec, exp, bits[t], dtype, f"t={t}")


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("dtype,block", [(0, 1), (0, 512), (0, 4096), (1, 64), (1, 2048), (2, 16), (2, 4096)])
def test_host_step_in_parts(dtype, block, pinned):
    """A step on host weights that is large enough to be cut into parts (pinned memory), with units of many sizes --
    their order in the tile table is not that of their addresses -- and long ones that straddle parts, also in the
    middle of a bitmap byte; twice in a row on the same plan.  Pageable memory: the step as a whole."""
    from paper_2609_04609_b200 import runtime

    sizes = [8192 * 40 + 3, 100, 0, 8192 * 200 + 4097, 8192 * 12 + 5, 1_000_000, 8192 * 3]
    codec = guard(runtime.LayerCodec.from_tensors(sizes, 1, NAME[dtype], block, DEV, slack=256))
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(3 * block + dtype)
    w = [wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    for _ in range(2):
        w.append(wl.step_clustered(w[-1], gen, f=0.3))
    bits = [wl.as_bits(x) for x in w]
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    staging = torch.empty(codec.weights_bytes, dtype=torch.uint8, device=DEV)
    wire_host = torch.zeros(codec.plan.n_units, dtype=torch.int64)
    for t in (1, 2):
        exp = table.step(bits[t])
        src = torch.from_numpy(bits[t].view(np.uint8).copy())
        out = torch.zeros(codec.weights_bytes, dtype=torch.uint8)
        if pinned:
            src, out, wire_host = src.pin_memory(), out.pin_memory(), wire_host.pin_memory()
        codec.step_host(src, out, staging, wire_host)
        torch.cuda.synchronize()
        codec.check_status()
        compare_step(codec, exp, bits[t], f"t={t}")
        compare_caches(codec, table, f"t={t}")
        compare_recon(codec, exp, bits[t], dtype, f"t={t}")
        assert np.array_equal(wire_host.numpy().astype(np.uint64), exp["wire"])
        assert torch.equal(staging.cpu(), src)
        host = out.numpy()
        for u in codec.units:
            lo, n = int(u["weights_off"]), int(u["n_values"]) * wl.VALUE_BYTES[NAME[dtype]]
            assert np.array_equal(host[lo : lo + n], src.numpy()[lo : lo + n])


@pytest.mark.parametrize("dtype,block", [(0, 512), (0, 4096), (1, 2), (2, 16)])
def test_long_runs_cut(dtype, block):
    """As many units of nine and ten tiles as the kernel has thread blocks: their runs of eight are handed out in pieces."""
    from paper_2609_04609_b200 import runtime

    sizes = [8192 * 10, 8192 * 9 + 1] * 148
    codec = guard(runtime.LayerCodec.from_tensors(sizes, 1, NAME[dtype], block, DEV, slack=256))
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(block + dtype, DEV)
    w = [wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    w += [wl.step_clustered(w[0], gen, f=0.3)]
    bits = [wl.as_bits(x) for x in w]
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    for t, step in ((1, three_calls), (0, one_launch)):
        exp = table.step(bits[t])
        step(codec, to_dev_bytes(bits[t], DEV))
        torch.cuda.synchronize()
        codec.check_status()
        compare_step(codec, exp, bits[t], f"t={t}")
        compare_caches(codec, table, f"t={t}")
        compare_recon(codec, exp, bits[t], dtype, f"t={t}")


@pytest.mark.parametrize("block", [1, 2, 8, 512])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_receiver_with_other_exponents_many_times(dtype, block):
    """The receiver's cache holds other exponents than the sender's, so that every reconstructed word differs from the
    weights it was staged with: a store that picks up the stage too early shows (fp32 leaves it by the copy engine)."""
    from paper_2609_04609_b200 import ciera, runtime

    one, three = (runtime.LayerCodec.from_tensors(SIZES, 1, NAME[dtype], block, DEV) for _ in range(2))
    gen = wl.make_generator(11 * block + dtype, DEV)
    n = one.weights_bytes // wl.VALUE_BYTES[NAME[dtype]]
    for rep in range(40):
        a = wl.init_weights(n, NAME[dtype], gen)
        b, other = wl.inject_exponent_changes(a, gen, 0.05), wl.init_weights(n, NAME[dtype], gen)
        for codec in (one, three):
            codec.init_caches(a.view(torch.uint8))
            ciera.cache_init(codec.plan, codec.receiver_cache, other.view(torch.uint8))
        one.step(b.view(torch.uint8))
        three_calls(three, b.view(torch.uint8))
        torch.cuda.synchronize()
        one.check_status()
        for u in one.units:
            lo = int(u["weights_off"])
            hi = lo + int(u["n_values"]) * wl.VALUE_BYTES[NAME[dtype]]
            assert torch.equal(one.weights_out[lo:hi], three.weights_out[lo:hi]), f"pass {rep}, values from {lo}"


@pytest.mark.parametrize("block", [1, 512])
@pytest.mark.parametrize("dtype", [0, 1, 2])
@pytest.mark.parametrize("where", ["weights - 64 KB", "weights + 16", "weights + 24 MB", "sent message"])
def test_output_over_buffers_that_thethree_calls_are_done_with(dtype, block, where):
    """Where the reconstructed weights go over bytes that the sender has read or sent by then, a step does what the three
    calls do: the message holds the weights as they were."""
    from paper_2609_04609_b200 import runtime

    codec = runtime.LayerCodec.from_tensors(SIZES + [8192 * 4000], 1, NAME[dtype], block, DEV)
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(17 * block + dtype)
    w0 = wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)
    bits = [wl.as_bits(x) for x in (w0, wl.step_clustered(w0, gen, f=0.3))]
    n = codec.weights_bytes
    room = torch.zeros(n + (25 << 20), dtype=torch.uint8, device=DEV)
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    w = room[1 << 17 :][:n]
    w.copy_(torch.from_numpy(bits[1].view(np.uint8)))
    if where == "sent message":
        codec.weights_out = codec.msg_send[:n]
    else:
        at = {"weights - 64 KB": -(1 << 16), "weights + 16": 16, "weights + 24 MB": 24 << 20}[where]
        codec.weights_out = room[(1 << 17) + at :][:n]
    exp = table.step(bits[1])
    codec.step(w)
    torch.cuda.synchronize()
    codec.check_status()
    if where == "sent message":
        codec.msg_send = codec.msg_recv  # (what was sent is gone; what arrived is compared twice)
    compare_step(codec, exp, bits[1], where)
    compare_caches(codec, table, where)
    compare_recon(codec, exp, bits[1], dtype, where)


@pytest.mark.parametrize("block", [1, 8, 16, 512])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_every_remainder_of_a_short_tile(dtype, block):
    """Units that end at every place of a 16-byte piece, in their first tile and in a later one, with bytes behind the last
    value that would count as changed exponents: sender, hashed sender and whole step."""
    from paper_2609_04609_b200 import runtime

    sizes = list(range(1, 35)) + [8192 + r for r in range(1, 17)] + [8192 * 3 + 500 + r for r in range(16)]
    codec = guard(runtime.LayerCodec.from_tensors(sizes, 1, NAME[dtype], block, DEV, slack=256))
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(13 * block + dtype)
    w = [wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    for _ in range(3):
        w.append(wl.inject_exponent_changes(w[-1], gen, 0.2))
    bits = [wl.as_bits(x).copy() for x in w]
    inside = np.zeros(bits[0].size, bool)
    for u in codec.units:
        lo = int(u["weights_off"]) // wl.VALUE_BYTES[NAME[dtype]]
        inside[lo : lo + int(u["n_values"])] = True
    for b in bits:
        b[~inside] = np.iinfo(b.dtype).max
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    guard(codec)  # (the bytes behind the cached exponents as well)
    if block >= 16:
        codec.init_hash_cache(to_dev_bytes(bits[0], DEV))
    for t, step in ((1, three_calls), (2, one_launch), (3, three_calls)):
        exp = table.step(bits[t])
        x = to_dev_bytes(bits[t], DEV)
        if block >= 16:  # the same message from the other sender, before the caches move on
            codec.encode_hashed(x)
            torch.cuda.synchronize()
            sent, wire = codec.msg_send.cpu().numpy(), codec.wire_bytes.tolist()
            assert wire == exp["wire"].tolist(), f"hashed t={t}"
            for u, n in zip(codec.units, wire):
                lo = int(u["msg_off"])
                assert np.array_equal(sent[lo : lo + n], exp["msgs"][lo : lo + n]), f"hashed t={t}"
        step(codec, x)
        torch.cuda.synchronize()
        codec.check_status()
        compare_step(codec, exp, bits[t], f"t={t}")
        compare_caches(codec, table, f"t={t}")
        compare_recon(codec, exp, bits[t], dtype, f"t={t}")


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_every_remainder_of_the_last_tile_of_a_buffer(dtype, shared):
    """The unit that ends the buffers, with every remainder and a different one for weights and caches; with ``shared``,
    two units have the same weights, so that several tiles end the weights buffer."""
    from paper_2609_04609_b200 import ciera, runtime

    vb, block = wl.VALUE_BYTES[NAME[dtype]], 16
    for n in list(range(1, 34)) + [8192 + r for r in range(1, 17)]:
        cap = ciera.message_capacity(n, dtype, block)
        slot = (cap + 15) // 16 * 16
        other = (n + 7) if not shared else n  # first in the caches, last in the weights (or in the same place there)
        rows = [(other, 0 if shared else (n * vb + 15) // 16 * 16, 0, 2 * slot + 64, ciera.message_capacity(other, dtype, block)),
                (n, 0, (other + 15) // 16 * 16, 0, cap)]
        units = np.array(rows, dtype=wl.UNIT_DTYPE)
        values = int(max(u["weights_off"] // vb + u["n_values"] for u in units))
        codec = runtime.LayerCodec(units, NAME[dtype], block, values * vb, int(rows[1][2]) + n, 5 * slot + 256, DEV, slack=256)
        table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
        gen = wl.make_generator(n + dtype)
        w = [wl.init_weights(values, NAME[dtype], gen)]
        for _ in range(2):
            w.append(wl.inject_exponent_changes(w[-1], gen, 0.3))
        bits = [wl.as_bits(x) for x in w]
        table.init_caches(bits[0])
        codec.init_caches(to_dev_bytes(bits[0], DEV))
        codec.allocations["sender_cache"][codec.cache_bytes :] = 0xEE
        codec.allocations["receiver_cache"][codec.cache_bytes :] = 0xEE
        room = torch.full((values * vb + 16,), 0xEE, dtype=torch.uint8, device=DEV)
        for t, step in ((1, three_calls), (2, one_launch)):
            exp = table.step(bits[t])
            room[: values * vb] = torch.from_numpy(bits[t].view(np.uint8).copy()).to(DEV)
            step(codec, room[: values * vb])
            torch.cuda.synchronize()
            codec.check_status()
            compare_step(codec, exp, bits[t], f"n={n} t={t}")
            compare_caches(codec, table, f"n={n} t={t}")
            compare_recon(codec, exp, bits[t], dtype, f"n={n} t={t}")


def test_small_tables_on_several_streams_beside_a_large_one():
    """Tables of a tile to a thread block (look-back between blocks that need not all be resident), of a few tiles to a
    block and of runs, stepped over and over on streams of their own while a large table keeps the SMs busy."""
    from paper_2609_04609_b200 import runtime

    gen = wl.make_generator(77, DEV)
    tables = [[524_288], [8192 * 250], [3_000_005, 131_072], [8192] * 40, [2_097_152] * 3, [8192 * 5 + 3] * 300, [8192 * 290 + 1], [4099]]
    jobs = []
    for i, sizes in enumerate(tables + [[2_097_152] * 48]):
        dtype = (0, 1, 2)[i % 3]
        codec = runtime.LayerCodec.from_tensors(sizes, 4, NAME[dtype], (512, 16, 1, 64)[i % 4], DEV)
        a = wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)
        w = [wl.step_clustered(a, gen, f=0.3).view(torch.uint8), a.view(torch.uint8)]
        codec.init_caches(w[1])
        jobs.append((codec, w, torch.cuda.Stream()))
    torch.cuda.synchronize()
    for it in range(60):
        for i, (codec, w, stream) in enumerate(jobs):
            for rep in range(1 if i == len(jobs) - 1 else 3):
                codec.step(w[(3 * it + rep) & 1 if i < len(jobs) - 1 else it & 1], None, stream)
    torch.cuda.synchronize()
    for i, (codec, w, _) in enumerate(jobs):
        codec.check_status()
        last = w[(3 * 59 + 2) & 1 if i < len(jobs) - 1 else 59 & 1]
        vb = wl.VALUE_BYTES[codec.dtype_name]
        for u in codec.units:
            lo, hi = int(u["weights_off"]), int(u["weights_off"]) + vb * int(u["n_values"])
            assert torch.equal(codec.weights_out[lo:hi], last[lo:hi]), f"table {i}"
        assert torch.equal(codec.sender_cache, codec.receiver_cache), f"table {i}"


def long_tiles_min(dtype):
    """Tiles of long units from which a whole step is run by the kernel instance for them, and how many a unit needs to be
    long, as the library has it."""
    src = os.path.join(os.path.dirname(__file__), "..", "paper_2609_04609_b200", "csrc", "ciera_internal.cuh")
    with open(src) as f:
        text = f.read()
    a, b = re.search(r"kLongTilesMin = (\d+) \* (\d+);", text).groups()
    least16 = re.search(r"kLongTilesMinFp16 = (\d+);", text).group(1)
    more16 = re.search(r"dtype == CIERA_FP16 \? (\d+)u : kSeqMaxTiles", text).group(1)
    return (int(least16), int(more16)) if dtype == 2 else (int(a) * int(b), 32)


def scratch_is_empty(codec):
    """The sender's words and all counters are handed back empty, whatever words the call laid out there."""
    return not codec.workspace[: 8 * codec.plan.n_tiles + 32].any()


@pytest.mark.parametrize("block", [16, 512, 4096])
@pytest.mark.parametrize("dtype", [0, 1, 2])
def test_tables_of_long_units(dtype, block):
    """Thousands of tiles in units of more than 32: units that start and end inside, and on the edge of, the groups of 32
    tiles whose words the look-back reads, ragged ends, and runs of short units beside them; hardly any, some and nearly all
    blocks changed; steps and the three calls, whose words are others, in turn on one scratch; once more in parts from host
    memory."""
    from paper_2609_04609_b200 import runtime

    tile = 8192
    shorts = [tile * 5] * 240 + [100] * 16  # (1216 tiles: the first long unit starts on the edge of a group)
    # starts on an edge; ends on one; both; ends inside; starts and ends inside, twice; ragged; ends on an edge
    tiles = [160 + 1, 191, 224, 163, 1024, 137, 5201, 1283] if dtype == 2 else [33, 63, 64, 35, 1024, 41, 2001, 323]
    longs = [tile * n for n in tiles]
    longs[3] -= 4097
    longs[5] -= 8189
    longs[6] -= 8115
    sizes = longs[:3] + shorts + longs[3:]
    assert [(n + tile - 1) // tile for n in longs] == tiles
    first = 1216 + np.concatenate([[0], np.cumsum(tiles)])  # (long units come behind the short ones in the tile table)
    assert [int(x) % 32 for x in first] == [0, 1, 0, 0, 3, 3, 12, 29, 0]
    least, more = long_tiles_min(dtype)
    assert sum(tiles) >= least and min(tiles) > more
    codec = guard(runtime.LayerCodec.from_tensors(sizes, 1, NAME[dtype], block, DEV, slack=256))
    assert codec.plan.n_tiles == first[-1]
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(17 * block + dtype, DEV)
    w = [wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    for model, kw in (("clustered", {"f": 0.3}), ("inject", {"c": 0.9}), ("inject", {"c": 1e-5}), ("clustered", {"f": 0.2})):
        step = wl.step_clustered if model == "clustered" else wl.inject_exponent_changes
        w.append(step(w[-1], gen, **kw))
    bits = [wl.as_bits(x) for x in w]
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    steps = ((1, one_launch), (2, three_calls), (3, one_launch), (4, None))
    for t, step in steps[1:] if dtype == 2 else steps:  # (the oracle takes its time over fp16)
        exp = table.step(bits[t])
        if step:
            step(codec, to_dev_bytes(bits[t], DEV))
        else:
            host = torch.from_numpy(bits[t].view(np.uint8).copy()).pin_memory()
            out = torch.zeros_like(host).pin_memory()
            codec.step_host(host, out, torch.empty(host.numel(), dtype=torch.uint8, device=DEV))
        torch.cuda.synchronize()
        codec.check_status()
        assert scratch_is_empty(codec), f"t={t}"
        compare_step(codec, exp, bits[t], f"t={t}")
        compare_caches(codec, table, f"t={t}")
        if step:
            compare_recon(codec, exp, bits[t], dtype, f"t={t}")
        else:
            for u in codec.units:
                lo, hi = (int(u["weights_off"]) + k * int(u["n_values"]) * wl.VALUE_BYTES[NAME[dtype]] for k in (0, 1))
                assert torch.equal(out[lo:hi], host[lo:hi])


@pytest.mark.parametrize("dtype,block", [(0, 16), (0, 4096), (1, 16), (2, 512)])
def test_long_units_beside_many_short_ones(dtype, block):
    """As many long tiles as the instance for long units asks for, but more in short units that it is slower with: the
    other instance steps them (see test_long_units_rule.py), with the three calls in turn on one scratch."""
    from paper_2609_04609_b200 import runtime

    tile = 8192
    codec = guard(runtime.LayerCodec.from_tensors([tile * 1300] + [1000] * 3000 + [tile * 1100 + 5], 1, NAME[dtype], block, DEV, slack=256))
    assert dtype == 2 or long_tiles_min(dtype)[0] <= 2401 < 3000
    table = OracleTable(codec.units, dtype, block, codec.cache_bytes, codec.msg_bytes)
    gen = wl.make_generator(19 * block + dtype, DEV)
    w = [wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[NAME[dtype]], NAME[dtype], gen)]
    for _ in range(2):
        w.append(wl.step_clustered(w[-1], gen, f=0.3))
    bits = [wl.as_bits(x) for x in w]
    table.init_caches(bits[0])
    codec.init_caches(to_dev_bytes(bits[0], DEV))
    for t, step in ((1, one_launch), (2, three_calls), (0, one_launch)):
        exp = table.step(bits[t])
        step(codec, to_dev_bytes(bits[t], DEV))
        torch.cuda.synchronize()
        codec.check_status()
        assert scratch_is_empty(codec), f"t={t}"
        compare_step(codec, exp, bits[t], f"t={t}")
        compare_caches(codec, table, f"t={t}")
        compare_recon(codec, exp, bits[t], dtype, f"t={t}")


@pytest.mark.parametrize("dtype,block", [(0, 512), (1, 64), (2, 16), (2, 4096)])
def test_long_units_in_place_from_a_graph_and_on_two_streams(dtype, block):
    """Two tables of long units stepped at once on streams of their own; then one of them replayed from a graph, and with
    the reconstructed weights put where the weights are: what the three calls make of the same weights."""
    from paper_2609_04609_b200 import runtime

    tile, vb = 8192, wl.VALUE_BYTES[NAME[dtype]]
    gen = wl.make_generator(29 * block + dtype, DEV)
    jobs = []
    for sizes in ([tile * 6000 + 5, tile * 2700], [tile * 3900, 77, tile * 4750 - 9]):
        assert sum(n // tile for n in sizes) >= long_tiles_min(dtype)[0]
        one, three = (runtime.LayerCodec.from_tensors(sizes, 1, NAME[dtype], block, DEV) for _ in range(2))
        w = [wl.init_weights(one.weights_bytes // vb, NAME[dtype], gen)]
        for _ in range(6):
            w.append(wl.step_clustered(w[-1], gen, f=0.3))
        w = [x.view(torch.uint8) for x in w]
        for codec in (one, three):
            codec.init_caches(w[0])
        jobs.append((one, three, w, torch.cuda.Stream()))
    torch.cuda.synchronize()

    def same(one, three, x, out, what):
        torch.cuda.synchronize()
        for codec in (one, three):
            codec.check_status()
        assert scratch_is_empty(one), what
        for name in ("sender_cache", "receiver_cache", "wire_bytes", "changed_blocks"):
            assert torch.equal(getattr(one, name), getattr(three, name)), f"{what}: {name}"
        for u, n in zip(one.units, one.wire_bytes.tolist()):
            lo, hi = int(u["weights_off"]), int(u["weights_off"]) + vb * int(u["n_values"])
            assert torch.equal(out[lo:hi], x[lo:hi]), f"{what}: values from {lo}"
            lo = int(u["msg_off"])
            for name in ("msg_send", "msg_recv"):
                assert torch.equal(getattr(one, name)[lo : lo + n], three.msg_send[lo : lo + n]), f"{what}: {name} from {lo}"

    for t in (1, 2, 3):
        for one, _, w, stream in jobs:
            one.step(w[t], None, stream)
    for one, three, w, _ in jobs:
        for t in (1, 2, 3):
            three_calls(three, w[t])
        same(one, three, w[3], one.weights_out, "two streams")
    one, three, w, _ = jobs[0]
    x = w[4].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        one.step(x)
    for t in (4, 5):
        x.copy_(w[t])
        graph.replay()
        three_calls(three, w[t])
        same(one, three, w[t], one.weights_out, "graph")
    x.copy_(w[6])
    one.step(x, x)
    three_calls(three, w[6])
    same(one, three, w[6], x, "in place")
