"""Parity of bf16 planes that are held in registers as they lie in memory (planes of 2,689 to 3,136 and of 4,481 to 5,376 groups of
four) with the oracle: at the edges of those ranges, on and off the 16-byte grid, and with values for which a threshold on distances is
hard to turn into one on elements.  How planes are held depends on how many there are: the first tests' few are held as fp32, the same
sizes and values come again in tests with as many as are held as words."""
import numpy as np
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity, gpu_compress, oracle_compress

pytestmark = pytest.mark.gpu

PLANES = [(1, 10752), (1, 10753), (127, 93), (104, 112), (1, 11651), (112, 112), (1, 12545), (1, 17920), (1, 17921), (139, 131), (1, 18305), (140, 140),
          (3, 6571), (88, 224), (1, 19713), (146, 146), (96, 224), (1, 21505)]


@pytest.mark.parametrize("hw", PLANES)
def test_parity_at_the_edges_of_the_ranges(hw):
    for bits, kind in ((2, "relu"), (4, "spiky_relu"), (8, "normal"), (4, "laplace_ch")):
        full_parity(synth.TensorSpec("t", (3, 17, *hw), synth.BF16, kind, 91), bits=bits)
    full_parity(synth.TensorSpec("t", (3, 17, *hw), synth.BF16, "normal", 92), bits=4, salient_mode=api.FH_SALIENT_OFF)
    full_parity(synth.TensorSpec("t", (3, 17, *hw), synth.BF16, "spiky_normal", 93), bits=2, rounding=1)


def values():
    """bf16 planes, as fp32, whose thresholds fall on hard elements: with the mean near the middle of a range that spans zero, so that
    lo + threshold cancels; subnormal; with both zeros; a few elements far off; steps of one unit in the last place."""
    rng = np.random.default_rng(94)
    n = 112 * 112
    spread = rng.standard_normal(n).astype(np.float32)
    small = spread * np.float32(1e-3)
    planes = [spread, -np.abs(spread), np.where(rng.random(n) < 0.01, np.float32(1.0), small), np.where(rng.random(n) < 0.01, np.float32(-1.0), small),
              small * np.float32(1e-36), np.select([spread > 1, spread > 0], [np.float32(0.0), np.float32(-0.0)], np.float32(-1.0)),
              np.where(rng.random(n) < 0.02, np.float32(-0.0), np.abs(small)), np.float32(1.0) + spread * np.float32(0.01),
              np.float32(-256.0) + spread, np.where(rng.random(n) < 0.005, np.float32(3e38), spread), np.full(n, 0.5, np.float32),
              np.round(spread), np.where(rng.random(n) < 0.03, spread * np.float32(1e-38), np.float32(-1.0) + small),
              np.where(rng.random(n) < 0.5, np.float32(1.0), np.float32(-1.0)) * np.exp(-8.0 * np.abs(spread)).astype(np.float32)]
    for t in range(3, 10):  # a rare value at about three sigma of the others, above and below a range around zero
        p = 1.0 / (t * t)
        planes.append(np.where(rng.random(n) < p, np.float32(1.0), small * np.float32(1e-4)))
        planes.append(np.where(rng.random(n) < p, np.float32(-1.0), small * np.float32(1e-4)))
    return np.stack(planes)


@pytest.mark.parametrize("bits", [2, 4, 8])
def test_parity_of_hard_thresholds(bits):
    x = values()
    raw = synth.to_bf16_bits(x.reshape(-1))
    shape = (1, x.shape[0], 112, 112)
    st_o, buf_o, total_o, _ = oracle_compress(raw, shape, synth.BF16, bits=bits)
    st_g, packed, total_g = gpu_compress(raw, shape, synth.BF16, bits=bits)
    assert st_o == st_g == api.FH_OK and total_o == total_g
    assert np.array_equal(packed[:total_g].cpu().numpy(), buf_o)


def room(hw):
    """Planes that are worked on at once, held as fp32 and as words (with three-sigma statistics): 20 and 24 warps to an SM."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    warps = -(-(-(-hw[0] * hw[1] // 4)) // 448)
    return sms * (20 // warps), sms * (24 // warps)


@pytest.mark.parametrize("hw", [hw for hw in PLANES if 10753 <= hw[0] * hw[1] <= 12544 or 17921 <= hw[0] * hw[1] <= 21504])
def test_parity_of_as_many_planes_as_are_held_as_words(hw):
    n = room(hw)[0] + 1
    full_parity(synth.TensorSpec("t", (1, n, *hw), synth.BF16, "laplace_ch", 95), bits=4)
    full_parity(synth.TensorSpec("t", (1, n, *hw), synth.BF16, "spiky_relu", 96), bits=2)
    full_parity(synth.TensorSpec("t", (1, n, *hw), synth.BF16, "normal", 97), bits=8, salient_mode=api.FH_SALIENT_OFF)
    full_parity(synth.TensorSpec("t", (1, n, *hw), synth.BF16, "spiky_normal", 98), bits=2, rounding=1)


@pytest.mark.parametrize("hw", [(112, 112), (134, 134), (146, 146)])
def test_parity_where_the_numbers_of_planes_change_how_they_are_held(hw):
    fp32, words = room(hw)
    for n in (1, fp32, words, words + 1, 5 * fp32, 5 * fp32 + 1):
        full_parity(synth.TensorSpec("t", (1, n, *hw), synth.BF16, "laplace_ch", 99), bits=2)


def test_parity_of_hard_thresholds_in_planes_held_as_words():
    x = np.tile(values(), (12, 1))
    raw = synth.to_bf16_bits(x.reshape(-1))
    shape = (1, x.shape[0], 112, 112)
    assert room((112, 112))[0] < x.shape[0] <= room((112, 112))[1]
    st_o, buf_o, total_o, _ = oracle_compress(raw, shape, synth.BF16, bits=4)
    st_g, packed, total_g = gpu_compress(raw, shape, synth.BF16, bits=4)
    assert st_o == st_g == api.FH_OK and total_o == total_g
    assert np.array_equal(packed[:total_g].cpu().numpy(), buf_o)
