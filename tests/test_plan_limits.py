"""Plans that neither tree kernel is meant to take are refused: a delay spread whose windows leave the direct
kernel little room (its widest windows run only where the leaf-sharing kernel would do) and whose leaf patterns
do not fit the leaf-sharing kernel. Host only."""
import numpy as np
import pytest

import paper_2606_15361_gb300 as g


def _plan(dm):
    freqs = 416.0 - (np.arange(768) + 0.5) * (16.0 / 768)
    return g.Plan(freqs, 1.38e-4, np.linspace(0.0, dm, 32), 64, g.MODE_FLOAT, g.options(g.MODE_FLOAT, max_chunk=8192),
                  bind=False)


def test_widest_windows():
    assert _plan(770.0).stats().tree_kernel == 1
    for dm in (790.0, 800.0, 840.0, 900.0):
        with pytest.raises(g.SndError, match="SND_ERR_UNSUPPORTED"):
            _plan(dm)
