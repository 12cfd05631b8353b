"""Tensor sizes that the benchmark prints, against the storage arithmetic
written out (here) and against the library's own count (on a GPU)."""
import numpy as np
import pytest

import bench
from paper_2107_05364_gb300 import workloads as wl


def _solid(nx, ny, nz):
    return wl.grid_tiles(np.linspace(0, nx * 5e-9, nx + 1), np.linspace(0, ny * 5e-9, ny + 1),
                         np.linspace(0, nz * 5e-9, nz + 1), 8e5, 1.3e-11, 0.0)


def test_dense_planes():
    film, solid = wl.film(50, 10, 1), _solid(10, 10, 5)  # 500 tiles: 512 rows and columns
    assert bench.mt_tensor_gb(film, "bf16") * 1e9 == pytest.approx(4 * 512 * 512 * 2)
    assert bench.mt_tensor_gb(film, "split") * 1e9 == pytest.approx(4 * 512 * 512 * 4)
    assert bench.mt_tensor_gb(solid, "bf16") * 1e9 == pytest.approx(6 * 512 * 512 * 2)


def test_streaming_planes():
    assert bench.mt_tensor_gb(wl.film(50, 40, 1), "f32") * 1e9 == pytest.approx(4 * 4 * 2000**2)
    assert bench.mt_tensor_gb(_solid(20, 10, 10), "f32") * 1e9 == pytest.approx(6 * 4 * 2000**2)
    # 6,400 tiles of one shape: three planes of the upper triangle (of 128-column chunks)
    assert bench.mt_tensor_gb(wl.film(160, 40, 1), "f32") * 1e9 == pytest.approx(3 * 4 * 50 * 51 / 2 * 128**2)
    graded = wl.graded_film(100, 50, 1, (500e-9, 250e-9, 3e-9), seed=1)
    assert bench.mt_tensor_gb(graded, "f32") * 1e9 == pytest.approx(4 * 4 * 5000**2)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["f32", "bf16", "split"])
def test_the_library_stores_as_much(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2107_05364_gb300 import build
    build.build()
    from paper_2107_05364_gb300 import binding as mt
    ctx = mt.mt_ctx_create(0)
    for t in (wl.film(128, 40, 1), _solid(16, 16, 20), _solid(16, 16, 8)):  # multiples of 128: no ragged chunk
        T = mt.mt_demag_assemble_ex(mt.mt_tiles_create(ctx, t), prec,
                                    mt.MT_LAYOUT_STREAM if prec == "f32" else mt.MT_LAYOUT_DENSE)
        assert T.info()["bytes"] == pytest.approx(bench.mt_tensor_gb(t, prec) * 1e9, rel=1e-9)
        T.close()
