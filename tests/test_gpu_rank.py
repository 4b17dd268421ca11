"""Blocks of an exact number of runs and islands around the lines where the candidate stage changes its
form: 2048 runs (islands joined) and 512 runs (candidates ranked by one CTA or the whole grid), 2048 keys a
shared-memory tile of the ranking, 256 candidates a CTA. Every channel fires at isolated samples of an
otherwise constant chunk, so a row has one run per sample, and equal trial DMs join their rows' runs.
Two blocks a plan (the second list is appended), alone and in a batch; lists equal the C++ oracle's."""
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

N, NCHAN = 48000, 8


def _chunk(islands, first):
    x = np.full((N, NCHAN), 100, dtype=np.uint8)
    x[first + 23 * np.arange(islands)] = 255
    return x


def _plan(ndm, flags=0):
    o = g.options(g.MODE_FLOAT, det_theta=3.5, closing_size=1, n_min_pixels=1, sigma_min=0.0, max_chunk=N, flags=flags)
    return g.Plan(synth.channel_freqs(NCHAN), synth.NC_DT, np.zeros(ndm), 2, g.MODE_FLOAT, o)


def _tuples(cands):
    return [(int(c["dm_index"]), int(c["t"]), float(c["snr"]), int(c["width"]), int(c["npix"])) for c in cands]


@pytest.mark.parametrize("reference", [False, True], ids=["cooperative", "staged"])
@pytest.mark.parametrize("ndm,islands", [(1, 1), (1, 255), (1, 256), (1, 257), (1, 511), (1, 512), (1, 513),
                                         (1, 2047), (1, 2048), (1, 2049), (2, 1024), (2, 1025), (3, 682), (3, 683),
                                         (5, 2060)])
def test_blocks_around_the_lines(ndm, islands, reference):
    chunks = [_chunk(islands, 300), _chunk(max(1, islands - 3), 57)]
    cfg = ostream.defaults(ostream.FLOAT, branching=2, det_theta=3.5, n_min=1, closing=1, sigma_min=0.0)
    ref = cxx.Stream(synth.channel_freqs(NCHAN), synth.NC_DT, np.zeros(ndm), cfg)
    exp = []
    for c in chunks:
        exp += [(k[0], k[2], float(k[3]), k[4], k[5]) for k in ref.push(c)["candidates"]]
    assert len(exp) == islands + max(1, islands - 3)
    flags = g.FLAG_REFERENCE_TREE if reference else 0
    one = _plan(ndm, flags)
    pair = [_plan(ndm, flags), _plan(ndm, flags)]
    batch = g.Batch(pair)
    for c in chunks:
        dev = torch.from_numpy(c).cuda()
        one.execute(dev)
        batch.execute([dev, dev])
    for p in [one] + pair:
        got, rc = p.candidates()
        assert rc == 0 and _tuples(got) == exp
