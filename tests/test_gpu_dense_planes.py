"""The batched tensor-core product over entry planes (6, or 4 for a single
layer) at the edges of its tiles: tile counts around the 64-column K block and
the 128-row tile, few units (fewer than SMs) and rows shared by many CTAs,
batch widths around each padded width, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2107_05364_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
TOL = {"bf16": 5e-3, "split": 1e-6}  # the precisions' stated field errors


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


@pytest.mark.parametrize("prec", ["bf16", "split"])
@pytest.mark.parametrize("shape,batches", [((1, 1, 1), (1,)), ((21, 3, 1), (2, 17)), ((16, 2, 2), (16,)),
                                           ((13, 5, 1), (33,)), ((127, 1, 1), (5, 65)), ((43, 3, 1), (64,)),
                                           ((13, 5, 2), (8, 128)), ((19, 9, 5), (1, 32, 64, 100))])
def test_field_matches_oracle(mt, ctx, prec, shape, batches):
    import torch
    nx, ny, nz = shape
    t = wl.graded_film(nx, ny, nz, (nx * 5e-9, ny * 5e-9, nz * 4e-9), seed=sum(shape))
    T = mt.mt_demag_assemble_ex(mt.mt_tiles_create(ctx, t), prec, mt.MT_LAYOUT_DENSE)
    assert T.info()["planes"] == (4 if nz == 1 else 6)
    model = oracle.Model.from_tiles(t)
    for B in batches:
        m = np.stack([wl.m_random(t.n, seed=7 * b + 1) for b in range(B)]).astype(np.float32)
        mg = torch.tensor(m.ravel(), device="cuda")
        H = torch.full_like(mg, float("nan"))
        for _ in range(2):  # the second call finds the counters as the first left them
            mt.mt_demag_field(T, mg, H, B)
        Hg = H.cpu().numpy().reshape(B, t.n, 3)
        for b in sorted({0, B // 2, B - 1}):
            ref = np.asarray(oracle.demag_field(model, m[b].astype(np.float64))).reshape(-1, 3)
            assert np.linalg.norm(Hg[b] - ref) <= TOL[prec] * np.linalg.norm(ref), (B, b)
        assert np.isfinite(Hg).all()
