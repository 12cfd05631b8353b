"""Selection and run storage of a thresholded tensor at the edges of the
32-column words, 128-column chunks and 4-row blocks that its kernels walk:
the same cut, kept elements and stored values as the oracle's selection on
the stored FP32 tensor (whole numbers and copies of values: no tolerance)."""
import numpy as np
import pytest

import oracle
from paper_2107_05364_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2107_05364_gb300 import build
    build.build()
    from paper_2107_05364_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(mt):
    return mt.mt_ctx_create(0)


def tiles(kind, n):
    # a line of equal tiles (many equal magnitudes: ties at the cut), a graded
    # two-layer strip (6 planes), a wide film (runs broken at every row of tiles)
    if kind == "line":
        return wl.film(n, 1, 1, size=(5e-9 * n, 5e-9, 3e-9))
    if kind == "layers":
        return wl.graded_film((n + 1) // 2, 1, 2, (4e-9 * n, 6e-9, 6e-9), seed=n)
    return wl.film(max(1, n // 9), 9, 1, size=(20e-9 * max(1, n // 9), 45e-9, 3e-9))


@pytest.mark.parametrize("kind", ["line", "layers", "film"])
@pytest.mark.parametrize("n", [1, 3, 31, 33, 127, 129, 260])
def test_selection_at_word_and_chunk_edges(mt, ctx, kind, n):
    t = tiles(kind, n)
    T = mt.mt_demag_assemble(mt.mt_tiles_create(ctx, t), "f32")
    N32 = mt.mt_tensor_read_rows(T, 0, t.n)
    for fraction in (0.0, 0.3, 0.85, 0.995):
        S, thr, kept = mt.mt_tensor_threshold(T, fraction)
        Nt, thr_o, kept_o = oracle.threshold_tensor(N32, fraction)
        assert np.float32(thr) == np.float32(thr_o) and kept == kept_o, fraction
        np.testing.assert_array_equal(mt.mt_tensor_read_rows(S, 0, t.n), Nt)
