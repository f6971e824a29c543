"""Decompression of small outlier-rich planes from payloads made by hand: consistent ones restore to the oracle's values, and
ones whose codes ask for more verbatim values than the payload holds are rejected."""
import numpy as np
import pytest

from oracle import fho
from paper_2510_11400_b200 import api, synth
from tests import helpers as hp
from tests.test_gpu_parity import check_same_values, to_dev

pytestmark = pytest.mark.gpu


def salient_container(shape, dtype, bits, codes, n_out_d, values):
    """A container whose planes all carry the same payload: its first block dense with `codes`, the others empty."""
    P, H, W = shape[0] * shape[1], shape[2], shape[3]
    d = fho.desc(shape, dtype)
    raw = np.zeros(P * H * W, dtype=np.float32 if dtype == synth.F32 else np.uint16)
    st, buf, total = fho.compress(raw, d, fho.params(bits=bits, salient_mode=fho.OFF))
    assert st == fho.OK
    word = np.uint32(values.nbytes + 3 & ~3)
    pay = np.concatenate([np.array([0, 1, n_out_d, 0, 1], np.uint32).view(np.uint8), np.zeros(4 * (H + 1), np.uint8),
                          codes.astype(np.uint8).reshape(-1), values.view(np.uint8), np.zeros(int(word) - values.nbytes, np.uint8)])
    pay = np.concatenate([pay, np.zeros(-pay.size % 16, np.uint8)])
    assert pay.size <= hp.a16(H * W * (4 if dtype == synth.F32 else 2))       # (or it would not be an outlier-rich plane's)
    npay, slots = hp.npay_of(buf, H * W), 64 + 16 * P
    over = pay[npay:]
    out = np.concatenate([buf[:slots + P * npay], np.zeros(P * over.size, np.uint8)])
    tab = out[64:slots].view(np.uint32).reshape(P, 4)
    tab[:] = 0
    tab[:, 1] = fho.SALIENT
    for p in range(P):
        out[slots + p * npay:slots + (p + 1) * npay][:pay.size] = pay[:npay]
        if over.size:
            off = slots + P * npay + p * over.size
            out[off:off + over.size] = over
            tab[p, 0] = off // 16
    out[40:44].view(np.uint32)[0] = P
    out[56:64].view(np.uint64)[0] = out.size
    return out, d


# planes of one block and of two to four, on and off the 16-byte grid; (verbatim values that fit the payload)
@pytest.mark.parametrize("shape,dtype,fit", [((1, 300, 5, 5), synth.F32, 1), ((1, 301, 8, 8), synth.BF16, 2), ((2, 65, 8, 8), synth.F32, 34),
                                             ((1, 300, 1, 24), synth.F32, 1), ((1, 37, 9, 8), synth.BF16, 2),
                                             ((1, 40, 16, 16), synth.F32, 64), ((1, 41, 15, 13), synth.BF16, 60)])
@pytest.mark.parametrize("bits", [2, 8])
def test_verbatim_values_of_small_planes(shape, dtype, fit, bits):
    H, W = shape[2:]
    inside = np.zeros((8, 8), bool)
    inside[:min(H, 8), :min(W, 8)] = True
    spots = np.flatnonzero(inside)
    rng = np.random.default_rng(3)
    fit = min(fit, spots.size)
    codes = np.full(64, 128, np.uint8)
    codes[spots] = rng.integers(120, 137, spots.size)
    codes[rng.choice(spots, fit, replace=False)] = 0
    values = synth.normal(fit, 4) if dtype == synth.F32 else synth.to_bf16_bits(synth.normal(fit, 4))
    buf, d = salient_container(shape, dtype, bits, codes, fit, np.ascontiguousarray(values))
    st_o, out_o = fho.decompress(buf, d)
    st_g, out_g = api.decompress_tensor(to_dev(buf), buf.size, shape, dtype)
    assert (st_o, st_g) == (fho.OK, api.FH_OK)
    got = out_g.cpu().numpy()
    check_same_values(got.view(np.uint16) if dtype == synth.BF16 else got, out_o, dtype)
    # one value fewer than the codes ask for, and codes that ask for 64 with none there
    for c, n in ((codes, fit - 1), (np.zeros(64, np.uint8), 0)):
        buf, d = salient_container(shape, dtype, bits, c, n, np.ascontiguousarray(values[:n]))
        assert fho.decompress(buf, d)[0] == fho.ERR_CORRUPT
        assert api.decompress_tensor(to_dev(buf), buf.size, shape, dtype)[0] == api.FH_ERR_CORRUPT
