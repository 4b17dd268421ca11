"""Reading candidates and destroying a plan wait for that plan's stream only: work of another stream, enqueued
before, is still running afterwards."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402
import synth  # noqa: E402


def _plan(mode, stream):
    with torch.cuda.stream(stream):
        return g.Plan(synth.channel_freqs(64), synth.NC_DT, synth.dm_grid(64, 50.0), 4, mode,
                      g.options(mode, max_chunk=2048), stream=stream)


def test_reads_and_destruction_do_not_wait_for_other_streams():
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    chunk = torch.from_numpy(np.full((2048, 64), 100, dtype=np.uint8)).cuda()
    plans = [_plan(g.MODE_FLOAT, mine) for _ in range(2)]
    torch.cuda.synchronize()
    a = torch.randn(4096, 4096, device="cuda")
    with torch.cuda.stream(other):
        b = a @ a  # kernels are loaded before the other stream is busy, which can wait for the GPU
    plans[1].execute(chunk, stream=mine)
    plans[1].candidates()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(other):
        for _ in range(200):  # more than 200 x 2 * 4096^3 / 1e14 = 0.27 s in FP32
            torch.mm(a, a, out=b)
        done.record()
    p = plans[0]
    p.execute(chunk, stream=mine)
    assert len(p.candidates()[0]) == 0
    g.lib.snd_destroy(p.handle)
    p.handle = None
    assert not done.query()  # the other stream's work outlives the plan
    torch.cuda.synchronize()
    del plans
