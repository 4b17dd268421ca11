"""Snippet standardisation at its edges against the FP64 oracle: snippets that hang over every
side of the plane, planes whose mean is far above their deviation, constant planes, deviations
outside the range of the FP32-pair arithmetic, infinities and NaN.

Tolerance: the result is the FP32 rounding (2^-24 relative) of a value whose mean, difference
and product carry about 45 bits, so 2^-23 of the value plus 2^-40 (1 + |mean| / deviation)."""
import numpy as np
import pytest

from oracle import sifter as osf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2606_15361_gb300 as g  # noqa: E402

ROWS = np.array([100, 0, 199, 31, 32, 168, 5, 190], dtype=np.int32)
COLS = np.array([700, 0, 1300, 127, 128, 1173, 1299, 3], dtype=np.int64)


def _plane(kind):
    rng = np.random.default_rng(21)
    x = rng.normal(size=(200, 1301)).astype(np.float32)
    return {"unit": x, "counts": np.rint(x * 8 + 68) / np.float32(32), "offset": x + np.float32(1e3),
            "far_offset": x + np.float32(1e6), "large": x * np.float32(1e12), "constant": np.full_like(x, 3.25),
            "tiny": x * np.float32(1e-30), "huge": x * np.float32(1e30),
            "one_inf": np.where(np.arange(x.size).reshape(x.shape) == 100 * 1301 + 700, np.float32(np.inf), x),
            "one_nan": np.where(np.arange(x.size).reshape(x.shape) == 100 * 1301 + 700, np.float32(np.nan), x),
            }[kind].astype(np.float32)


@pytest.mark.parametrize("kind", ["unit", "counts", "offset", "far_offset", "large", "constant", "tiny", "huge",
                                  "one_inf", "one_nan"])
def test_snippets_at_the_edges(kind):
    plane = _plane(kind)
    # a plane view with a row pitch above its width
    dp = torch.zeros((200, 1400), dtype=torch.float32, device="cuda")[:, :1301]
    dp.copy_(torch.from_numpy(plane))
    out = g.snippets(dp, torch.from_numpy(ROWS).cuda(), torch.from_numpy(COLS).cuda()).cpu().numpy()
    for i in range(len(ROWS)):
        with np.errstate(all="ignore"):
            exp = osf.snippet(plane, int(ROWS[i]), int(COLS[i]))
        fin = np.isfinite(exp)
        assert np.array_equal(fin, np.isfinite(out[i])) and np.array_equal(np.isnan(exp), np.isnan(out[i]))
        cells = plane.astype(np.float64)[max(0, ROWS[i] - 32):ROWS[i] + 32, max(0, COLS[i] - 128):COLS[i] + 128]
        with np.errstate(all="ignore"):
            sd = cells.std()
            ratio = abs(cells.mean()) / sd if np.isfinite(sd) and sd > 0 else 0.0
        tol = 2.0 ** -23 * np.abs(exp[fin]) + 2.0 ** -40 * (1.0 + ratio)
        assert np.all(np.abs(out[i][fin].astype(np.float64) - exp[fin]) <= tol), kind
