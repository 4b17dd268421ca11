"""The one-launch encoder at its edges: chunk lengths around ring words and cluster shares, chunks that
start inside a word, one-sample chunks, channel counts and chunk addresses that allow 16-, 4- and
1-byte loads, degenerate channels, and a chunk too long for it (the three-kernel form). The spikes are
seen through the float planes of trial DMs with different delays per channel; their counts are
integers and must be equal."""
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

DMS = np.array([0.0, 3.0, 11.0, 40.0])


def _chunk(rng, n, nchan):
    x = np.clip(np.rint(rng.normal(128, 16, (n, nchan))), 0, 255).astype(np.uint8)
    x[:, 0] = 77                                   # constant: never fires
    if nchan > 3:
        x[:, 1] = np.where(rng.random(n) < 0.02, 255, 0)   # two values, the rare one clipped
        x[:, 2] = rng.integers(0, 256, n)          # uniform over all 256 values
        x[:, 3] = 255
    return x


@pytest.mark.parametrize("batch", [False, True], ids=["single", "batch"])
@pytest.mark.parametrize("nchan,offset,lengths", [
    (64, 0, [1, 31, 32, 33, 1, 2000, 255, 256, 257, 4097]),
    (48, 0, [3000, 8192, 5]),
    (64, 4, [777, 2049]),          # 4-byte loads by address
    (36, 0, [777, 2049, 640]),     # 4-byte loads by channel count, a block of four channels
    (33, 0, [1500, 64, 2500]),     # byte loads, a block of one channel
    (64, 1, [1500, 3001]),         # byte loads by address
    (7, 0, [900, 900]),
    (64, 0, [50000, 300]),         # the first chunk is too long for shared memory
])
def test_spikes_equal_the_oracle(nchan, offset, lengths, batch):
    rng = np.random.default_rng(5)
    freqs = synth.channel_freqs(nchan)
    theta = 0.75
    # a wider detection threshold keeps the candidate list out of the way; chunks stay below the limit
    o = g.options(g.MODE_FLOAT, enc_theta=theta, det_theta=1e6, max_chunk=max(lengths))
    plan = g.Plan(freqs, synth.NC_DT, DMS, 4, g.MODE_FLOAT, o)
    step = g.Batch([plan]) if batch else None
    delay = odelays.delay_table(freqs, synth.NC_DT, DMS)
    spikes, done = np.zeros((nchan, 0), dtype=np.int64), 0
    for n in lengths:
        x = _chunk(rng, n, nchan)
        buf = torch.zeros(n * nchan + offset, dtype=torch.uint8, device="cuda")
        dev = buf[offset:].view(n, nchan)
        dev.copy_(torch.from_numpy(x))
        spikes = np.concatenate([spikes, oenc.encode_chunk(x, theta)[0].astype(np.int64)], axis=1)
        ne = plan.nemit_next(n)
        if batch:
            step.execute([dev])
            out = None
        else:
            out = torch.full((len(DMS), max(ne, 1)), -1.0, dtype=torch.float32, device="cuda")
            assert plan.execute(dev, out) == ne
        if ne and out is not None:
            exp = np.stack([sum(spikes[c, done + delay[d, c]:done + delay[d, c] + ne] for c in range(nchan))
                            for d in range(len(DMS))])
            got = np.rint(out[:, :ne].cpu().numpy().astype(np.float64) * np.sqrt(nchan)).astype(np.int64)
            assert np.array_equal(got, exp)
        done += ne
    assert plan.candidates()[1] == 0
    if batch:  # the ring the batch filled gives the same plane of a further chunk
        x = _chunk(rng, 700 if max(lengths) >= 700 else max(lengths), nchan)
        spikes = np.concatenate([spikes, oenc.encode_chunk(x, theta)[0].astype(np.int64)], axis=1)
        ne = plan.nemit_next(len(x))
        out = torch.full((len(DMS), max(ne, 1)), -1.0, dtype=torch.float32, device="cuda")
        plan.execute(torch.from_numpy(x).cuda(), out)
        exp = np.stack([sum(spikes[c, done + delay[d, c]:done + delay[d, c] + ne] for c in range(nchan))
                        for d in range(len(DMS))])
        assert np.array_equal(np.rint(out[:, :ne].cpu().numpy().astype(np.float64) * np.sqrt(nchan)).astype(np.int64), exp)
