"""Which tables the whole step runs with its instance for long units (``runs_as_long_units`` in ``csrc/ciera_internal.cuh``):
not those in which short units that this instance is slower with outweigh the long ones.  On the CPU."""
import os
import subprocess

import pytest

from paper_2609_04609_b200.build import _nvcc

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.join(HERE, "..")
BF16, FP32, FP16 = 0, 1, 2
LEAST = {BF16: 8 * 296, FP32: 8 * 296, FP16: 8192}


@pytest.fixture(scope="module")
def chosen(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("long_units") / "long_units_rule")
    subprocess.run([_nvcc(), "-std=c++17", "-x", "cu", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2609_04609_b200", "csrc"), os.path.join(HERE, "long_units_rule.cpp"), "-o", exe], check=True)

    def ask(dtype, block, longs, others=0, ragged=0):
        line = f"{dtype} {block.bit_length() - 1} {longs} {others} {ragged}\n"
        return bool(int(subprocess.run([exe], input=line, check=True, capture_output=True, text=True).stdout))

    return ask


@pytest.mark.parametrize("dtype", [BF16, FP32, FP16])
@pytest.mark.parametrize("block", [16, 32, 64, 128, 512, 4096])
def test_long_units_alone(chosen, dtype, block):
    assert not chosen(dtype, block, LEAST[dtype] - 1)
    assert chosen(dtype, block, LEAST[dtype]) == (dtype != FP16 or block not in (32, 64))


# tiles of long units, other tiles, ragged ones among them, and what such a table took by the other instance / by this one, us
@pytest.mark.parametrize("dtype,block,longs,others,ragged,want", [
    (BF16, 512, 21504, 98664, 360, True),      # fine-grained experts and dense tensors: 1783 / 1753
    (BF16, 512, 4096, 196608, 196608, False),  # units of 1024 values: 1299 / 1522
    (FP32, 512, 4096, 196608, 196608, False),  # 2026 / 3041
    (FP16, 512, 8192, 196608, 196608, False),
    (BF16, 16, 4096, 49152, 0, True),          # a layer: 615 / 603
    (FP32, 32, 4096, 24576, 0, True),          # half a layer: 654 / 638
    (FP32, 16, 4096, 24576, 0, False),         # 676 / 790
    (FP32, 16, 16384, 24576, 0, False),        # 1031 / 1099
    (FP32, 16, 8192, 0, 0, True),              # 248 / 224
    (FP16, 64, 16384, 49152, 0, False),        # 877 / 888
    (FP16, 512, 8192, 2048, 1024, False),      # units of 9001 values: 169.1 / 170.9
    (FP16, 512, 8192, 4096, 0, True),          # 197.4 / 190.4
])
def test_other_units_beside_long_ones(chosen, dtype, block, longs, others, ragged, want):
    assert chosen(dtype, block, longs, others, ragged) == want
