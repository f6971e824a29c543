"""Parity with the oracle where many outlier-rich planes are put off: more tiles or planes than a CTA of the warp-team kernel
lists, planes that pass through the queue of the CTA-team kernels (measurements kept in the slot, with and without the
Huffman code, or too large for it), statistics over channels in pieces and over many small planes, from call to call."""
import numpy as np
import pytest

from oracle import fho
from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity, to_dev

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


def test_parity_of_overlapping_calls_on_two_streams():
    """Kernels with planes put off on two streams at once, each with more CTAs than find room beside the other's: every call
    must come through with the bytes of a call alone."""
    import torch
    calls, p = [], api.default_params(bits=4, salient_mode=api.FH_SALIENT_ALL)
    for i, (shape, dtype) in enumerate([((2, 350, 112, 112), synth.BF16), ((2, 700, 56, 56), synth.F32)]):
        raw = synth.make(synth.TensorSpec("t", shape, dtype, "spiky_relu", 43 + i))
        st, buf, total = fho.compress(raw, fho.desc(shape, dtype), fho.params(bits=4, salient_mode=fho.ALL))
        assert st == fho.OK
        d = api.desc(shape, dtype)
        dst = [torch.zeros(api.compressed_bytes(d, p, 1), dtype=torch.uint8, device="cuda") for _ in range(6)]
        calls.append((to_dev(raw), d, buf, total, dst, torch.zeros(6, 2, dtype=torch.int64, device="cuda"), torch.cuda.Stream()))
    torch.cuda.synchronize()
    for k in range(6):
        for x, d, _, _, dst, out2, stream in calls:
            assert api.fh_compress(d, p, x, dst[k], out2[k], stream=stream) == api.FH_OK
    torch.cuda.synchronize()
    for _, _, buf, total, dst, out2, _ in calls:
        want = to_dev(buf)
        assert out2.tolist() == [[total, api.FH_OK]] * 6
        assert all(torch.equal(t[:total], want) for t in dst)


@pytest.mark.parametrize("mode", [api.FH_SALIENT_CHANNEL, api.FH_SALIENT_TENSOR])
@pytest.mark.parametrize("shape", [(4, 6, 28, 28), (2, 5000, 7, 7)])   # statistics cleared by the call itself, and ahead of the next
def test_channel_statistics_of_a_captured_call(mode, shape):
    """A captured call starts from cleared statistics each time it is replayed, and so do calls made in between."""
    import torch
    rng = np.random.default_rng(45)   # (no outliers in uniform draws)
    raws = [scale * rng.random(int(np.prod(shape)), dtype=np.float32) for scale in (np.float32(1), np.float32(-3))]
    want = [to_dev(fho.compress(r, fho.desc(shape), fho.params(bits=4, salient_mode=mode))[1]) for r in raws]
    assert all(fho.parse_header(w.cpu().numpy())["n_salient"] == 0 for w in want)
    xs = [to_dev(r) for r in raws]
    p, d = api.default_params(bits=4, salient_mode=mode), api.desc(shape)
    x, dst = torch.empty_like(xs[0]), torch.zeros(api.compressed_bytes(d, p, 1), dtype=torch.uint8, device="cuda")
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        x.copy_(xs[0])
        assert api.fh_compress(d, p, x, dst) == api.FH_OK
        with torch.cuda.graph(graph, stream=stream):
            assert api.fh_compress(d, p, x, dst) == api.FH_OK
        for k in (0, 1, 1, 0):
            x.copy_(xs[k])
            for step in (graph.replay, graph.replay, lambda: api.fh_compress(d, p, x, dst)):
                dst.zero_()
                step()
                assert torch.equal(dst[:want[k].numel()], want[k])
    torch.cuda.synchronize()


# fewer rows of blocks than the team has warps: the rows are measured and written in parts
@pytest.mark.parametrize("shape", [(2, 20, 1, 5000), (1, 12, 8, 1001), (1, 12, 17, 700), (1, 20, 3, 1100), (1, 6, 40, 880)])
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
@pytest.mark.parametrize("entropy", [0, 1])
def test_parity_of_flat_planes(shape, dtype, entropy):
    full_parity(synth.TensorSpec("t", shape, dtype, "spiky_relu", 46), bits=4, entropy=entropy, salient_mode=api.FH_SALIENT_ALL)
    full_parity(synth.TensorSpec("t", shape, dtype, "spiky_normal", 47), bits=2, entropy=entropy, eps=0.25)


def test_schedules_of_two_host_threads_on_one_stream():
    """The workspace a stream keeps for the next schedule goes to one caller at a time; schedules of different lengths."""
    import threading
    import torch
    stream, p = torch.cuda.Stream(), api.default_params(bits=4)
    jobs = []
    for t, count in enumerate((3, 400)):
        shape = (2, 16, 14, 14)
        raws = [to_dev(synth.make(synth.TensorSpec("s", shape, synth.F32, "spiky_relu", 800 + 10 * t + i % 3))) for i in range(count)]
        items = [api.SchedItem(api.desc(shape, tensor_id=i), api.FH_COMPRESS, x, torch.empty_like(x)) for i, x in enumerate(raws)]
        arena = torch.zeros(count * ((api.compressed_bytes(items[0].desc, p, 1) + 255) & ~255), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        rep = api.fh_run_schedule(items, p, arena, stream=stream)
        assert rep.status == api.FH_OK
        jobs.append((items, arena, rep.total_packed_bytes, arena.clone(), [i.restored.clone() for i in items]))
    torch.cuda.synchronize()
    bad = []

    def work(items, arena, packed, want, restored):
        for _ in range(20):
            arena.zero_()
            items[0].restored.zero_()
            torch.cuda.synchronize()
            rep = api.fh_run_schedule(items, p, arena, stream=stream)
            if (rep.status, rep.total_packed_bytes) != (api.FH_OK, packed) or not torch.equal(arena, want) or \
                    not all(torch.equal(i.restored, r) for i, r in zip(items, restored)):
                bad.append(len(items))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
