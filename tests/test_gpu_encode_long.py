"""Chunks around the longest that the one-launch encoder holds in shared memory (1512 ring words: 48,384
samples from a word's start) and the longest before its limit counted a CTA's static shared memory (1560
words), from a word's start and from inside a word: the spikes are seen through the float planes of two
trial DMs, whose counts are integers and must be equal. The larger one's sweep is about as long as a chunk,
so the second chunk's plane shows the whole of the first, which the batch encodes without a plane."""
import numpy as np
import pytest

import synth
from oracle import delays as odelays
from oracle import encoder as oenc

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402

DMS = np.array([0.0] * 32 + [3300.0])  # a 32-DM tile each
THETA = 0.75


@pytest.mark.parametrize("batch", [False, True], ids=["single", "batch"])
@pytest.mark.parametrize("nchan", [64, 33])
@pytest.mark.parametrize("before", [0, 5])
@pytest.mark.parametrize("n", [48379, 48380, 48384, 48385, 49152, 49920, 49921])
def test_spikes_of_the_longest_chunks(n, before, nchan, batch):
    rng = np.random.default_rng(n + before)
    freqs = synth.channel_freqs(nchan)
    # no detection reaches this threshold: the candidate list stays empty
    o = g.options(g.MODE_FLOAT, enc_theta=THETA, det_theta=1e6, max_chunk=n)
    plan = g.Plan(freqs, synth.NC_DT, DMS, 4, g.MODE_FLOAT, o)
    step = g.Batch([plan]) if batch else None
    delay = odelays.delay_table(freqs, synth.NC_DT, DMS)
    spikes, done = np.zeros((nchan, 0), dtype=np.int64), 0
    lengths = ([before] if before else []) + [n, n]
    for k, length in enumerate(lengths):
        x = np.clip(np.rint(rng.normal(128, 16, (length, nchan))), 0, 255).astype(np.uint8)
        x[::50, 1] = 255  # clipped
        spikes = np.concatenate([spikes, oenc.encode_chunk(x, THETA)[0].astype(np.int64)], axis=1)
        ne = plan.nemit_next(length)
        dev = torch.from_numpy(x).cuda()
        out = None
        if batch and k < len(lengths) - 1:
            step.execute([dev])  # seen in the plane of the last chunk
        else:
            out = torch.full((len(DMS), max(ne, 1)), -1.0, dtype=torch.float32, device="cuda")
            assert plan.execute(dev, out) == ne
        if ne and out is not None:
            got = np.rint(out[:, :ne].cpu().numpy().astype(np.float64) * np.sqrt(nchan)).astype(np.int64)
            for d in (0, 32):
                exp = sum(spikes[c, done + delay[d, c]:done + delay[d, c] + ne] for c in range(nchan))
                assert np.array_equal(got[d], exp)
            assert (got[1:32] == got[0]).all()
        done += ne
    assert plan.candidates()[1] == 0


@pytest.mark.parametrize("lengths", [
    (14592, 14593, 22272, 22273),                  # few CTAs: the beams of more than 14,592 samples in one launch
    (14592, 14593, 22272, 22273, 22273, 20000),    # more than the GPU takes one per SM: a launch per class
])
def test_batch_of_every_class(lengths):
    """Beams on both sides of the lines between three, two and one CTA per SM."""
    nchan, rng = 160, np.random.default_rng(len(lengths))
    freqs = synth.channel_freqs(nchan)
    plans, spikes, devs, delays = [], [], [], []
    for n in lengths:
        dms = DMS * (n / 47000.0)  # a sweep of about a chunk
        delays.append(odelays.delay_table(freqs, synth.NC_DT, dms))
        plans.append(g.Plan(freqs, synth.NC_DT, dms, 4, g.MODE_FLOAT,
                            g.options(g.MODE_FLOAT, enc_theta=THETA, det_theta=1e6, max_chunk=n)))
        x = [np.clip(np.rint(rng.normal(128, 16, (n, nchan))), 0, 255).astype(np.uint8) for _ in range(2)]
        spikes.append(np.concatenate([oenc.encode_chunk(c, THETA)[0].astype(np.int64) for c in x], axis=1))
        devs.append([torch.from_numpy(c).cuda() for c in x])
    done = [p.nemit_next(n) for p, n in zip(plans, lengths)]
    g.Batch(plans).execute([d[0] for d in devs])
    for p, n, s, d, t, delay in zip(plans, lengths, spikes, devs, done, delays):
        ne = p.nemit_next(n)
        out = torch.full((len(DMS), max(ne, 1)), -1.0, dtype=torch.float32, device="cuda")
        assert p.execute(d[1], out) == ne
        got = np.rint(out[:, :ne].cpu().numpy().astype(np.float64) * np.sqrt(nchan)).astype(np.int64)
        for r in (0, 32):
            assert np.array_equal(got[r], sum(s[c, t + delay[r, c]:t + delay[r, c] + ne] for c in range(nchan)))
        assert p.candidates()[1] == 0
