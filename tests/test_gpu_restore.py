"""Parity of the streaming decompress kernels with the oracle at the edges of their chunks (1,024 elements), on and off the 16-byte
grid, with normal, raw and outlier-rich planes, and of fp32 tensors beyond the L2 cache, which have a kernel of their own."""
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity

pytestmark = pytest.mark.gpu

PLANES = [(1, 513), (3, 171), (8, 65), (27, 19), (24, 24), (1, 1023), (32, 32), (25, 41), (1, 1028), (36, 57), (1, 2047), (64, 32),
          (23, 89), (1, 2056), (48, 64), (45, 47), (40, 40)]


@pytest.mark.parametrize("hw", PLANES)
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
def test_parity_at_the_edges_of_the_chunks(hw, dtype):
    for bits, kind in ((2, "relu"), (4, "spiky_relu"), (8, "normal")):
        full_parity(synth.TensorSpec("t", (3, 37, *hw), dtype, kind, 51), bits=bits)
    # mostly raw planes: nothing shrinks when every residual is too large for a code
    full_parity(synth.TensorSpec("t", (3, 37, *hw), dtype, "normal", 52), bits=4, eps=1e-5, salient_mode=api.FH_SALIENT_ALL)


@pytest.mark.parametrize("shape", [(34, 64, 128, 128), (35, 64, 127, 125), (175, 64, 57, 55), (1072, 64, 1, 513)])   # more than 128 MiB
@pytest.mark.parametrize("bits", [2, 8])
def test_parity_of_fp32_tensors_beyond_the_l2_cache(shape, bits):
    full_parity(synth.TensorSpec("t", shape, synth.F32, "spiky_relu", 53), bits=bits)


def test_parity_of_raw_planes_beyond_the_l2_cache():
    full_parity(synth.TensorSpec("t", (70, 64, 90, 91), synth.F32, "normal", 54), bits=2, eps=1e-5, salient_mode=api.FH_SALIENT_ALL)
