"""The receiver's counts of changed blocks before each tile, made segment by segment (``prefix_segment`` in
``csrc/ciera_internal.cuh``): units that end on and one value past the edges of a segment, with the smallest segments
and with longer ones (more than 32 of the smallest), against the weights that were sent; tolerance 0."""
import pytest
import torch

from harness import guard
from paper_2609_04609_b200 import workloads as wl

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
TILE = 8192


@pytest.mark.parametrize("tiles", [1, 15, 16, 17, 32, 255, 256, 257, 512, 513, 1030])
@pytest.mark.parametrize("dtype,block", [("bf16", 1), ("bf16", 16), ("fp16", 2), ("fp16", 32), ("fp32", 8), ("fp32", 16)])
def test_units_at_the_edges_of_segments(tiles, dtype, block):
    from paper_2609_04609_b200 import runtime

    codec = guard(runtime.LayerCodec.from_tensors([tiles * TILE, tiles * TILE + 1, 5 * TILE], 1, dtype, block, DEV, slack=256))
    gen = wl.make_generator(3 * tiles + block, DEV)
    w0 = wl.init_weights(codec.weights_bytes // wl.VALUE_BYTES[dtype], dtype, gen)
    w1 = wl.inject_exponent_changes(w0, gen, 0.3 / block)
    dev = [w.view(torch.uint8) for w in (w0, w1)]
    codec.init_caches(dev[0])
    for t in (1, 0):
        codec.encode(dev[t])
        codec.transport()
        codec.decode()
        torch.cuda.synchronize()
        codec.check_status()
        codec.canaries.check("segments")
        spans = [(int(u["weights_off"]), int(u["weights_off"]) + int(u["n_values"]) * wl.VALUE_BYTES[dtype]) for u in codec.units]
        for lo, hi in spans:
            assert torch.equal(codec.weights_out[lo:hi], dev[t][lo:hi])
        assert torch.equal(codec.receiver_cache, codec.sender_cache)
