"""Plans of several threads, each on its own stream, with chunks whose kernels need very different amounts of
shared memory: the candidates of every thread equal those of the same plan run alone."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402

# channels, chunk, DM span
BEAMS = [(64, 48000, 50.0), (64, 1000, 300.0), (128, 20000, 5.0), (100, 3000, 100.0)]
STEPS = 200


def _run(beam, chunk, stream, out, errors):
    nchan, n, span = beam
    try:
        torch.cuda.set_device(0)
        p = g.Plan(synth.channel_freqs(nchan), synth.NC_DT, np.linspace(0.0, span, 40), 4, g.MODE_FLOAT,
                   g.options(g.MODE_FLOAT, max_chunk=n, det_theta=5.0), stream=stream)
        for k in range(STEPS):
            p.execute(chunk, stream=stream)
            if k % 20 == 19:
                out.append(p.candidates()[0])
    except Exception as e:  # noqa: BLE001
        errors.append((beam, repr(e)))


def test_threads_do_not_disturb_one_another():
    rng = np.random.default_rng(3)
    chunks = [torch.from_numpy(np.clip(np.rint(rng.normal(128, 16, (n, c))), 0, 255).astype(np.uint8)).cuda()
              for c, n, _ in BEAMS]
    torch.cuda.synchronize()
    alone, together, errors = [[] for _ in BEAMS], [[] for _ in BEAMS], []
    for b, c, o in zip(BEAMS, chunks, alone):
        _run(b, c, torch.cuda.Stream(), o, errors)
    assert not errors
    threads = [threading.Thread(target=_run, args=(b, c, torch.cuda.Stream(), o, errors))
               for b, c, o in zip(BEAMS, chunks, together)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for a, b in zip(alone, together):
        assert len(a) == len(b) and all((x == y).all() for x, y in zip(a, b))
