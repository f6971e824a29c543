"""Parity of the streaming kernels with the oracle where their tiling changes: plane sizes on both sides of every change of
team, slots per lane, warps per CTA and kernel, planes that start off the 16-byte grid, tensors that end off it."""
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity

pytestmark = pytest.mark.gpu

# (h, w): a team of lanes per plane (4 elements to a group, 7 or 8 groups to a lane)
SMALL = [(1, 1), (1, 15), (4, 4), (1, 17), (4, 8), (3, 11), (7, 8), (1, 61), (8, 8), (1, 65), (7, 16), (11, 11), (1, 113),
         (16, 16), (5, 89), (7, 64), (16, 31), (23, 39), (31, 33), (32, 32)]
# a CTA per plane: warps of 225 to 448 groups, 10, 12, 13 or 14 slots to a lane
LARGE = [(13, 79), (32, 33), (37, 35), (33, 47), (31, 53), (40, 42), (32, 56), (43, 42), (43, 43), (56, 56), (59, 61), (64, 64), (73, 73),
         (112, 112), (113, 111), (149, 149)]


@pytest.mark.parametrize("hw", SMALL + LARGE)
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
def test_parity_at_the_edges_of_the_sweep(hw, dtype):
    shape = (1, 19, *hw)
    full_parity(synth.TensorSpec("t", shape, dtype, "normal", 31), bits=2)
    full_parity(synth.TensorSpec("t", shape, dtype, "spiky_relu", 32), bits=4)
    full_parity(synth.TensorSpec("t", shape, dtype, "relu", 33), bits=8, rounding=1, seed=99)
    full_parity(synth.TensorSpec("t", shape, dtype, "relu", 34), bits=8, salient_mode=api.FH_SALIENT_OFF)


# the first and the last plane size of five, six and seven slots to a lane, teams of 2, 8 and 32 lanes
SLOTS = [(1, 33), (5, 8), (1, 41), (6, 8), (7, 7), (1, 56), (3, 43), (10, 16), (7, 23), (12, 16), (1, 193), (14, 16),
         (27, 19), (20, 32), (1, 641), (24, 32), (1, 769), (28, 32)]


@pytest.mark.parametrize("hw", SLOTS)
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
def test_parity_at_the_edges_of_the_slots(hw, dtype):
    shape = (1, 23, *hw)
    full_parity(synth.TensorSpec("t", shape, dtype, "normal", 41), bits=4)
    full_parity(synth.TensorSpec("t", shape, dtype, "spiky_relu", 42), bits=2, rounding=1, seed=5)
    full_parity(synth.TensorSpec("t", shape, dtype, "relu", 43), bits=8, salient_mode=api.FH_SALIENT_ALL)


@pytest.mark.parametrize("hw", [(128, 280), (191, 187), (160, 228), (191, 191)])  # 35,840 elements and beyond: other kernels
def test_parity_beyond_the_register_kernel(hw):
    full_parity(synth.TensorSpec("t", (1, 3, *hw), synth.BF16, "spiky_relu", 35), bits=4)


# planes beyond the register kernel in fp32 (the general-purpose kernel), and the widest and tallest that fit
@pytest.mark.parametrize("hw,dtype", [((160, 228), synth.F32), ((191, 187), synth.F32), ((224, 224), synth.F32), ((1, 50614), synth.F32),
                                      ((2, 35544), synth.BF16), ((30000, 1), synth.BF16), ((300, 300), synth.BF16)])
def test_parity_of_the_largest_planes(hw, dtype):
    full_parity(synth.TensorSpec("t", (1, 9, *hw), dtype, "spiky_relu", 36), bits=2)
    full_parity(synth.TensorSpec("t", (1, 9, *hw), dtype, "relu", 37), bits=2, rounding=1, seed=7)
