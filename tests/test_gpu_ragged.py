"""The direct tree on channel counts that are not whole 64-channel groups (the rest are zero ring
rows), against the C++ oracle: planes and candidates as in test_gpu_direct, for ragged last leaves,
in-group nodes, top levels and exact-level nodes of every mode."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import test_gpu_direct as direct  # noqa: E402

B_, G_, F_ = direct.B_, direct.G_, direct.F_

CASES = [
    # name, nchan, B, ndm, dm_max, mode, kl, ki, cap, expect_direct
    ("float-1000-b8", 1000, 8, 70, 900.0, F_, 0, 0, 255, True),
    ("float-61-b2", 61, 2, 33, 80.0, F_, 0, 0, 255, True),
    ("float-2047-b4", 2047, 4, 32, 300.0, F_, 0, 0, 255, True),
    ("graded-1000-b8", 1000, 8, 40, 600.0, G_, 0, 0, 255, True),
    ("graded-1023-b8-cap100", 1023, 8, 40, 600.0, G_, 0, 0, 100, True),
    ("graded-640-b4", 640, 4, 31, 300.0, G_, 0, 0, 255, True),
    ("graded-701-b2-u2", 701, 2, 31, 300.0, G_, 0, 0, 255, True),
    ("graded-1280-b4-u2", 1280, 4, 31, 300.0, G_, 0, 0, 255, True),
    ("graded-250-root", 250, 8, 45, 200.0, G_, 0, 0, 255, True),
    ("graded-1010-b16-root", 1010, 16, 40, 600.0, G_, 0, 0, 255, True),
    ("binary-1000-b8-k2", 1000, 8, 64, 900.0, B_, 2, 2, 255, True),
    ("binary-1001-b8-k1", 1001, 8, 33, 600.0, B_, 1, 1, 255, True),
    ("binary-934-b4-k2", 934, 4, 33, 600.0, B_, 2, 2, 255, True),
    ("binary-700-b2-k1", 700, 2, 33, 300.0, B_, 2, 1, 255, True),
    ("binary-511-b8-k2", 511, 8, 33, 200.0, B_, 2, 2, 255, True),
    ("binary-185-b3-k1", 185, 3, 33, 200.0, B_, 1, 1, 255, True),
    ("binary-3950-b2-k1", 3950, 2, 32, 200.0, B_, 1, 1, 255, True),
    ("float-5-few", 5, 2, 20, 80.0, F_, 0, 0, 255, True),
]


@pytest.mark.parametrize("case", CASES, ids=[c[0] for c in CASES])
def test_ragged_channel_counts(case):
    direct.test_direct_kernel_cases(case)
