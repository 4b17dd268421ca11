"""The pattern-sharing labelled-payload tree at its edges, bit for bit against the oracle (every
addition and rounding is in the oracle's order, so there is no tolerance): calls that end just
before, at and after a time tile, DM counts around the 16-DM tile, trees of every depth class,
leaves of other sizes and a ragged last leaf, DM grids out of order with duplicates, ascending
frequencies, grids so coarse that no patterns are shared, and a tree of one leaf (the direct form)."""
import numpy as np
import pytest

import synth
from oracle import zpayload as oz

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402

# nchan, C, B, DM grid, emitted samples of the last call
CASES = {
    "tile_minus_1": (64, 4, 4, np.linspace(0, 30, 17), 767),
    "tile": (64, 4, 4, np.linspace(0, 30, 16), 768),
    "tile_plus_1": (64, 4, 4, np.linspace(0, 30, 15), 769),
    "many_tiles": (64, 4, 8, np.linspace(0, 20, 33), 5003),
    "one_sample": (64, 4, 8, np.linspace(0, 20, 3), 1),
    "two_levels": (24, 6, 4, np.linspace(0, 60, 20), 700),
    "six_levels": (128, 4, 2, np.linspace(0, 60, 20), 1500),
    "ten_levels": (512, 1, 2, np.linspace(0, 20, 18), 900),
    "eleven_levels": (1024, 1, 2, np.linspace(0, 10, 9), 300),
    "ragged_leaf": (101, 7, 3, np.linspace(0, 50, 19), 1300),
    "unsorted_dms": (64, 4, 4, np.array([9.0, 3.0, 3.0, 27.5, 0.0, 9.1, 14.0, 9.0, 30.0, 1.0, 2.0, 3.0, 8.0, 8.1, 7.9,
                                         22.0, 21.0, 30.0]), 1100),
    "one_leaf": (4, 4, 4, np.linspace(0, 300, 18), 900),
    "coarse": (64, 2, 4, np.linspace(0, 500, 16), 600),
}


@pytest.mark.parametrize("fp16", [True, False], ids=["fp16", "fp32"])
@pytest.mark.parametrize("name", list(CASES) + ["ascending"])
def test_planes_equal_the_oracle(name, fp16):
    nchan, C, B, dms, last = CASES["tile_plus_1" if name == "ascending" else name]
    freqs = synth.channel_freqs(nchan)
    if name == "ascending":
        freqs = freqs[::-1].copy()
    o = g.options(g.MODE_ZFLOAT, cluster_size=C, flags=g.FLAG_FP16_PARTIALS if fp16 else 0, max_chunk=45000)
    plan = g.Plan(freqs, synth.NC_DT, dms, B, g.MODE_ZFLOAT, o)
    ref = oz.ZStream(freqs, synth.NC_DT, dms, C, B, 1.5, np.float16 if fp16 else np.float32)
    rng = np.random.default_rng(17)
    for n in (plan.stats().max_delay + 37, last):
        chunk = np.clip(np.rint(rng.normal(128, 16, (n, nchan))), 0, 255).astype(np.uint8)
        ne = plan.nemit_next(n)
        out = torch.full((len(dms), max(ne, 1)), float("nan"), dtype=torch.float32, device="cuda")
        assert plan.execute(torch.from_numpy(chunk).cuda(), out) == ne
        exp = ref.push(chunk)["plane"]
        assert np.array_equal(out.cpu().numpy().view(np.uint32), exp.view(np.uint32))
    assert plan.candidates()[1] == 0
