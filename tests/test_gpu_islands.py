"""Islands of blocks with few and many runs, which are joined by one CTA in shared memory or by the whole
grid: low detection thresholds and small closing elements make blocks of thousands of runs. Single plans
and a batch whose beams differ; candidate lists equal the C++ oracle's."""
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

W = synth.NC64
# detection threshold, closing side, smallest island
CASES = [(2.5, 1, 1), (3.0, 1, 1), (3.0, 3, 2), (3.5, 9, 1), (4.0, 1, 1), (5.0, 3, 1), (7.0, 9, 10)]


def _plan(theta, closing, n_min, max_chunk):
    o = g.options(g.MODE_FLOAT, det_theta=theta, closing_size=closing, n_min_pixels=n_min, max_chunk=max_chunk)
    return g.Plan(W.freqs(), synth.NC_DT, W.dms(), 2, g.MODE_FLOAT, o)


def _expected(theta, closing, n_min, chunks):
    cfg = ostream.defaults(ostream.FLOAT, branching=2, det_theta=theta, n_min=n_min, closing=closing)
    ref = cxx.Stream(W.freqs(), synth.NC_DT, W.dms(), cfg)
    out = []
    for c in chunks:
        out += ref.push(c)["candidates"]
    return [(c[0], c[2], float(c[3]), c[4], c[5]) for c in out]


def _tuples(cands):
    return [(int(c["dm_index"]), int(c["t"]), float(c["snr"]), int(c["width"]), int(c["npix"])) for c in cands]


def test_islands_of_small_and_large_blocks():
    data = W.chunk_data(0)
    chunks = [data[:9000], data[9000:]]
    lengths = []
    plans = []
    for theta, closing, n_min in CASES:
        p = _plan(theta, closing, n_min, 9000)
        for c in chunks:
            p.execute(torch.from_numpy(np.ascontiguousarray(c)).cuda())
        got, rc = p.candidates()
        exp = _expected(theta, closing, n_min, chunks)
        assert rc == 0 and _tuples(got) == exp
        lengths.append(len(exp))
        plans.append((_plan(theta, closing, n_min, 9000), exp))
    assert max(lengths) > 4096 and min(lengths) < 100
    for group in (plans[:2], plans[4:], plans):  # all large, all small, mixed
        beams = [(_plan(*CASES[plans.index(q)], 9000), q[1]) for q in group]
        batch = g.Batch([b[0] for b in beams])
        for c in chunks:
            dev = torch.from_numpy(np.ascontiguousarray(c)).cuda()
            batch.execute([dev] * len(beams))
        for p, exp in beams:
            got, rc = p.candidates()
            assert rc == 0 and _tuples(got) == exp
