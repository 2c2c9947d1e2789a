"""The integer FP64 coarse apply with one vector per chirality (18 rows: one warp, fewer threads
than the words it clears for a group of four right-hand sides), against the stored blocks and, right-hand side
by right-hand side, against the launch for one; fields of different magnitudes, so that a maximum left
over from another group shows."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed_coarse import _apply, _check, _hierarchy, mg  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [2, 4, 12, 64])
def test_one_vector_per_chirality(mg, nrhs):  # noqa: F811
    s, A = _hierarchy(mg, 16, 8, 1)
    with s:
        x = W.gaussian_field((nrhs, 2, 2, 2), 3)
        x *= 2.0 ** (200 - 40 * (np.arange(nrhs) // 4 % 10))[:, None, None, None]
        y = _apply(mg, s, x)
        _check(A, x, y)
        for r in range(nrhs):
            assert np.array_equal(_apply(mg, s, x[r:r + 1].copy())[0], y[r])
