"""The rounded means a multi-rate step computes for its bands (whole words of four channels up to S = 256,
single bytes otherwise) equal oracle.multirate.scrunch byte for byte. Whole numbers: the bytes are equal or the
test fails. The staged rows are looked for in the bound workspace."""
import numpy as np
import pytest

import synth
from oracle import multirate as omr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402


@pytest.mark.parametrize("nchan,nsamp,offset", [(64, 8192, 0), (64, 512, 0), (62, 2048, 0), (68, 2048, 1), (4, 1024, 0),
                                                (1000, 2048, 0), (1028, 1536, 0), (1100, 2048, 2)])
def test_staged_rows_are_the_rounded_means(nchan, nsamp, offset):
    f = synth.channel_freqs(nchan)
    df, fc = abs(f[1] - f[0]), 0.5 * (f.max() + f.min())
    want = [1, 2, 4, 8, 16, 64, 128, 256, 512]
    dms = [1.2 * s * synth.NC_DT * fc ** 3 / (synth.K_SKY * df) for s in want]
    o = g.options(0, max_chunk=8192, cand_capacity=4096)
    plan = g.MultiRatePlan(f, synth.NC_DT, dms, 2, 0, o, s_max=512)
    assert plan.scrunch == want
    rng = np.random.default_rng(nchan + nsamp)
    x = rng.integers(0, 256, (nsamp, nchan), dtype=np.uint8)
    x[: nsamp // 2, : nchan // 2] = 255  # the largest sums
    d = torch.empty(nsamp * nchan + 16, dtype=torch.uint8, device="cuda")
    chunk = d[offset: offset + nsamp * nchan].view(nsamp, nchan)
    chunk.copy_(torch.from_numpy(x))
    plan.execute(chunk)
    torch.cuda.synchronize()
    ws = plan.workspace.cpu().numpy().tobytes()
    for s in want[1:]:
        assert ws.find(omr.scrunch(x, s).tobytes()) >= 0, s
