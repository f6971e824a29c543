"""Parity with the oracle where planes of more than four blocks are listed first and measured when the CTA has run out of tiles:
tiles that still lie in their stages and tiles that are fetched again, more planes than the list holds (32 to a CTA), several tiles
to a CTA whose places one warp looks up together, small tiles for the Huffman stage."""
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity

pytestmark = pytest.mark.gpu

ALL = dict(salient_mode=api.FH_SALIENT_ALL)
CASES = [
    ((1, 16, 28, 28), synth.F32, "spiky_relu", dict(bits=4)),               # one plane in all, its tile in its stage
    ((1, 33, 17, 17), synth.BF16, "spiky_relu", dict(bits=2, **ALL)),       # every plane, fewer than the list holds
    ((40, 192, 28, 28), synth.BF16, "spiky_relu", dict(bits=2)),            # two and three tiles to a CTA
    ((160, 192, 28, 28), synth.F32, "spiky_relu", dict(bits=8)),            # more tiles than stages: planes are fetched again
    ((96, 192, 17, 17), synth.F32, "spiky_normal", dict(bits=4)),           # ... off the 16-byte grid
    ((40, 192, 32, 32), synth.BF16, "spiky_relu", dict(bits=4, **ALL)),     # more planes than the list holds
    ((7, 999, 1, 40), synth.F32, "spiky_relu", dict(bits=4)),               # flat planes, two lanes to a plane
    ((3, 700, 1, 40), synth.BF16, "spiky_relu", dict(bits=8, **ALL)),
    ((1, 32, 7, 7), synth.F32, "spiky_relu", dict(bits=4, entropy=1)),
    ((8, 512, 7, 7), synth.F32, "spiky_relu", dict(bits=4, entropy=1)),
    ((8, 513, 7, 7), synth.BF16, "spiky_relu", dict(bits=2, entropy=1)),
    ((3, 100, 7, 7), synth.F32, "spiky_relu", dict(bits=8, entropy=1, **ALL)),
    ((64, 256, 14, 14), synth.F32, "spiky_relu", dict(bits=4, entropy=1)),
    ((2, 40, 1, 3), synth.F32, "spiky_relu", dict(bits=2, entropy=1, **ALL)),
]


@pytest.mark.parametrize("shape,dtype,kind,kw", CASES)
def test_parity_with_planes_measured_late(shape, dtype, kind, kw):
    full_parity(synth.TensorSpec("t", shape, dtype, kind, 48), **kw)


# small planes, several tiles to a CTA: places for all of a CTA's tiles at once, in stages and fetched again
@pytest.mark.parametrize("shape,dtype", [((40, 960, 7, 7), synth.BF16), ((300, 960, 7, 7), synth.BF16), ((100, 512, 8, 8), synth.F32),
                                         ((60, 512, 14, 14), synth.F32), ((200, 512, 4, 4), synth.F32)])
def test_parity_of_small_planes_in_many_tiles(shape, dtype):
    full_parity(synth.TensorSpec("t", shape, dtype, "relu", 49), bits=2)
    full_parity(synth.TensorSpec("t", shape, dtype, "spiky_relu", 50), bits=4)


# planes that are many in their slice of a tile, which are measured where they are found: tiles with only such planes, in their stages
# and fetched again; more of them than are listed; tiles of both kinds
@pytest.mark.parametrize("shape,dtype,kind,kw", [
    ((3333, 3, 54, 1), synth.BF16, "relu", dict(bits=2)),
    ((250, 128, 2, 43), synth.F32, "laplace_ch", dict(bits=4)),
    ((61, 24, 1, 89), synth.F32, "spiky_relu", dict(bits=8, **ALL)),
    ((300, 16, 172, 2), synth.F32, "spiky_relu", dict(bits=8, **ALL)),
    ((64, 64, 20, 20), synth.BF16, "spiky_relu", dict(bits=4, **ALL)),
    ((300, 999, 1, 40), synth.F32, "relu", dict(bits=4, **ALL)),
    ((300, 999, 1, 40), synth.BF16, "spiky_relu", dict(bits=2)),
    ((400, 61, 8, 3), synth.F32, "normal", dict(bits=4, entropy=1)),
    ((100000, 1, 1, 40), synth.F32, "spiky_relu", dict(bits=4)),            # all of them, two tiles to a CTA: more planes than are listed
    ((15000, 8, 1, 520), synth.BF16, "spiky_relu", dict(bits=2)),           # one in a tile, more tiles to a CTA than are listed
])
def test_parity_with_many_planes_in_a_slice(shape, dtype, kind, kw):
    full_parity(synth.TensorSpec("t", shape, dtype, kind, 51), **kw)


# Huffman stage, fewer tiles than SMs: tiles of eight, four, two planes and one, so that a warp's part of the stages holds less than a
# plane; on either side of each change
@pytest.mark.parametrize("planes", [147, 148, 294, 296, 297, 588, 592, 1176, 1184, 1185])
def test_parity_of_small_tiles(planes):
    full_parity(synth.TensorSpec("t", (1, planes, 32, 32), synth.F32, "spiky_relu", 52), bits=4, entropy=1, **ALL)
    full_parity(synth.TensorSpec("t", (1, planes, 31, 29), synth.BF16, "spiky_relu", 53), bits=2, entropy=1)
