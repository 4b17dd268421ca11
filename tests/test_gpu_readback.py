"""Candidate read-back around the head of the list that comes in one piece (512 candidates): lists
shorter and longer than it, caps below and above it, and a read on another stream's plan after a
reset. The candidates are exact, so the lists must be equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402
import synth  # noqa: E402


def _plan(capacity):
    o = g.options(g.MODE_FLOAT, det_theta=3.0, n_min_pixels=1, closing_size=1, max_chunk=16384, cand_capacity=capacity)
    return g.Plan(synth.channel_freqs(64), synth.NC_DT, synth.dm_grid(128, 100.0), 2, g.MODE_FLOAT, o)


def test_lists_past_the_head_come_back_whole():
    rng = np.random.default_rng(3)
    chunk = torch.from_numpy(np.clip(np.rint(rng.normal(128, 16, (16384, 64))), 0, 255).astype(np.uint8)).cuda()
    p = _plan(65536)
    p.execute(chunk)
    full, rc = p.candidates()
    assert rc == 0 and len(full) > 1100
    key = full["t"].astype(np.int64) * 128 + full["dm_index"]
    assert (np.diff(key) > 0).all()
    assert len(p.candidates()[0]) == 0  # the list was reset
    for cap in (0, 1, 511, 512, 513, 1000, len(full), len(full) + 1):
        q = _plan(65536)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        q.execute(chunk, stream=stream)
        got, rc = q.candidates(cap=cap, check=False)
        assert rc == (0 if cap >= len(full) else g.ERR["SND_ERR_OVERFLOW"])
        assert (got == full[:cap]).all() and len(got) == min(cap, len(full))
        q.execute(chunk)  # the reset holds for work on any stream
        assert q.candidates(check=False)[1] == 0
    for capacity in (1, 512, 600):
        q = _plan(capacity)
        q.execute(chunk)
        got, rc = q.candidates(check=False)
        assert rc == g.ERR["SND_ERR_OVERFLOW"] and len(got) <= capacity
