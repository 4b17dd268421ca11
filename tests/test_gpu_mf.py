"""The matched filter over row lengths of every launch shape (256, 512 and 1024 threads, one row per SM
and many), block starts at every offset from a 16-byte boundary, ring wraps, and blocks of a few start
times, in all modes and plane types: planes and candidates equal the C++ oracle's."""
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

# ndm, chunk lengths (the first fills the delays), plane dtype
CASES = [
    ("few_rows_short", 24, [2600, 1, 2, 3, 4, 5, 130, 127, 1000], 0),
    ("few_rows_long", 24, [2600, 5003, 17001, 16385, 20000], 0),
    ("few_rows_longest", 5, [2600, 40000, 41999], 0),
    ("many_rows_short", 400, [2600, 33, 4001, 4096, 999], 1),
    ("many_rows_mid", 400, [2600, 8001, 7999], 0),
    ("many_rows_long", 400, [2600, 16387, 16001], 0),
    ("many_rows_1024", 330, [2600, 33001, 30000], 1),
    ("many_rows_longest", 330, [2600, 42000, 41001], 0),
]


@pytest.mark.parametrize("mode", [ostream.BINARY, ostream.GRADED, ostream.FLOAT], ids=["binary", "graded", "float"])
@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_rows_of_every_shape(case, mode):
    name, ndm, lengths, dtype = case
    freqs, dms = synth.channel_freqs(64), np.linspace(0.0, 180.0, ndm)
    seed = 100 + len(name) + ndm
    n = sum(lengths)
    rng = np.random.default_rng(seed)
    bursts = [synth.Burst(float(t), float(rng.uniform(20, 170)), float(rng.uniform(2, 30)), float(rng.uniform(20, 60)))
              for t in np.linspace(200, n - 3200, 6)]
    data = synth.filterbank_chunk(seed, 0, 0, n, freqs, synth.NC_DT, bursts)
    o = g.options(mode, max_chunk=max(lengths))
    if dtype and mode != ostream.FLOAT:
        o.plane_dtype = 1
    plan = g.Plan(freqs, synth.NC_DT, dms, 4, mode, o)
    ref = cxx.Stream(freqs, synth.NC_DT, dms, ostream.defaults(mode, branching=4))
    exp_c, at = [], 0
    for k in lengths:
        ch = np.ascontiguousarray(data[at:at + k])
        at += k
        ne = plan.nemit_next(k)
        tt = torch.float32 if mode == ostream.FLOAT else (torch.uint8 if o.plane_dtype else torch.int32)
        out = torch.zeros((ndm, max(ne, 1)), dtype=tt, device="cuda")
        assert plan.execute(torch.from_numpy(ch).cuda(), out) == ne
        r = ref.push(ch)
        if ne:
            got = out[:, :ne].cpu().numpy()
            if mode == ostream.FLOAT:
                assert np.array_equal(np.rint(got.astype(np.float64) * 8.0), r["plane"])
            else:
                assert np.array_equal(got, r["plane"])
        exp_c += r["candidates"]
    got_c, rc = plan.candidates()
    assert rc == 0
    assert [(int(c["dm_index"]), int(c["t"]), float(c["snr"]), int(c["width"]), int(c["npix"])) for c in got_c] == \
        [(c[0], c[2], float(c[3]), c[4], c[5]) for c in exp_c]
