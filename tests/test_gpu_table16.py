"""The direct tree's 16-bit table entries, which serve DM grids so coarse that two CTAs per SM leave no room for
32-bit ones: windows on both sides of both lines, in every mode, alone and in a
batch with a 32-bit plan, with per-level fire counts; planes and candidates equal the C++ oracle's."""
import numpy as np
import pytest

import synth
from oracle import cxx
from oracle import stream as ostream

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402

CHUNK, NDM = 4096, 40
# channels, DM span of 32 trial DMs, dynamic shared memory of the tree: the widest 32-bit windows that fit, the
# narrowest and widest 16-bit ones, and 32-bit ones past those (one CTA per SM; 64 channels a round)
CASES = [(64, 356.0, 114944), (64, 364.0, 108800), (64, 392.0, 114944), (64, 400.0, 125184), (100, 364.0, 109056),
         (256, 364.0, 109568), (256, 92.0, 111616), (256, 96.0, 58368)]


def _dms(span):
    return np.linspace(0.0, span * (NDM - 1) / 31, NDM)


def _data(nchan, span):
    n = 4 * CHUNK
    bursts = [synth.Burst(float(t), float(0.9 * span * k / 4), 4.0, 40.0) for k, t in enumerate((300, 1500, 2900, 4000))]
    return synth.filterbank_chunk(nchan, 0, 0, n, synth.channel_freqs(nchan), synth.NC_DT, bursts)


def _plan(nchan, span, mode, B, **kw):
    return g.Plan(synth.channel_freqs(nchan), synth.NC_DT, _dms(span), B, mode, g.options(mode, max_chunk=CHUNK, **kw))


def _theta(mode):
    return {} if mode != ostream.BINARY else {"enc_theta": 0.5}  # quorums that fire


def _tuples(cands):
    return [(int(c["dm_index"]), int(c["t"]), float(c["snr"]), int(c["width"]), int(c["npix"])) for c in cands]


@pytest.mark.parametrize("mode,B", [(ostream.FLOAT, 2), (ostream.GRADED, 8), (ostream.BINARY, 8), (ostream.BINARY, 3)],
                         ids=["float", "graded", "binary8", "binary3"])
@pytest.mark.parametrize("nchan,span,smem", CASES)
def test_planes_and_candidates(nchan, span, smem, mode, B):
    data = _data(nchan, span)
    kw = _theta(mode)
    plan, pair = _plan(nchan, span, mode, B, **kw), [_plan(nchan, span, mode, B, **kw), _plan(nchan, 20.0, mode, B, **kw)]
    assert plan.stats().tree_kernel == 1 and plan.stats().tree_smem_bytes == smem
    batch = g.Batch(pair)
    refs = [cxx.Stream(synth.channel_freqs(nchan), synth.NC_DT, d, ostream.defaults(mode, branching=B, **kw))
            for d in (_dms(span), _dms(20.0))]
    exp = [[], []]
    for i in range(0, len(data), CHUNK):
        ch = np.ascontiguousarray(data[i:i + CHUNK])
        dev = torch.from_numpy(ch).cuda()
        ne = plan.nemit_next(CHUNK)
        out = torch.zeros((NDM, max(ne, 1)), dtype=torch.float32 if mode == ostream.FLOAT else torch.int32, device="cuda")
        assert plan.execute(dev, out) == ne
        batch.execute([dev, dev])
        r = [s.push(ch) for s in refs]
        if ne:
            got = out[:, :ne].cpu().numpy()
            if mode == ostream.FLOAT:
                got = np.rint(got.astype(np.float64) * np.sqrt(nchan))
            assert np.array_equal(got, r[0]["plane"])
        for k in (0, 1):
            exp[k] += [(c[0], c[2], float(c[3]), c[4], c[5]) for c in r[k]["candidates"]]
    for p, e in ((plan, exp[0]), (pair[0], exp[0]), (pair[1], exp[1])):
        got, rc = p.candidates()
        assert rc == 0 and _tuples(got) == e


@pytest.mark.parametrize("nchan,span", [(64, 392.0), (256, 364.0)])
def test_level_rates(nchan, span):
    """Fire counts do not depend on the tile: 16-bit entries with 8 warps, 32-bit ones with 4."""
    data = torch.from_numpy(_data(nchan, span)).cuda()
    fires = []
    for warps in (0, 4):
        p = _plan(nchan, span, g.MODE_FLOAT, 4, flags=g.FLAG_LEVEL_RATES, tree_warps=warps)
        for i in range(0, len(data), CHUNK):
            p.execute(data[i:i + CHUNK])
        fires.append(p.level_rates()[0])
    assert (fires[0] == fires[1]).all() and fires[0][0] > 0
