"""Parity with the oracle where many outlier-rich planes are put off: more tiles or planes than a CTA of the warp-team kernel
lists, planes that pass through the queue of the CTA-team kernels (measurements kept in the slot, with and without the
Huffman code, or too large for it), statistics over channels in pieces and over many small planes, from call to call."""
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity

pytestmark = pytest.mark.gpu

CASES = [
    # a tile of 256 planes, more than 32 tiles to a CTA (3 CTAs on each of 148 SMs)
    ((4, 950000, 2, 2), synth.BF16, "normal", dict(bits=2)),
    # a tile of 32 planes of six blocks, more than 128 planes to a CTA
    ((8, 9001, 17, 9), synth.F32, "spiky_relu", dict(bits=4)),
    ((3, 700, 40, 41), synth.BF16, "spiky_relu", dict(bits=2)),
    ((3, 700, 56, 56), synth.F32, "spiky_relu", dict(bits=8)),
    ((2, 400, 56, 56), synth.F32, "spiky_relu", dict(bits=4, entropy=1)),
    ((2, 400, 56, 56), synth.F32, "spiky_relu", dict(bits=2, entropy=1)),
    ((2, 900, 28, 28), synth.BF16, "spiky_relu", dict(bits=8, entropy=1)),
]


@pytest.mark.parametrize("shape,dtype,kind,kw", CASES)
def test_parity_with_every_plane_put_off(shape, dtype, kind, kw):
    full_parity(synth.TensorSpec("t", shape, dtype, kind, 41), salient_mode=api.FH_SALIENT_ALL, **kw)


@pytest.mark.parametrize("mode", [api.FH_SALIENT_CHANNEL, api.FH_SALIENT_TENSOR])
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
def test_parity_of_channel_statistics(mode, dtype):
    for shape in [(5, 3, 150, 151), (3, 700, 3, 3), (4, 33, 64, 72), (2, 17, 45, 47), (9, 1, 1, 1), (3, 700, 8, 8)]:
        full_parity(synth.TensorSpec("t", shape, dtype, "spiky_relu", 42), bits=4, salient_mode=mode)
