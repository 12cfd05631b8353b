"""The batched product where its CTAs' ranges change: one row tile (one CTA),
the first tile of a second one, ranges of four units that end inside row tiles
and K blocks, and the size from which every SM has a range.  Against the FP64
oracle, and the same bits on a second call."""
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


@pytest.mark.parametrize("prec", ["bf16", "split"])
@pytest.mark.parametrize("shape,batches", [((8, 1, 1), (33, 128)), ((16, 8, 1), (16, 65)), ((8, 8, 2), (33,)),
                                           ((43, 3, 1), (33,)), ((25, 14, 1), (4, 128)), ((7, 7, 8), (33, 64)),
                                           ((9, 9, 9), (12, 33))])
def test_field_matches_oracle(mt, prec, shape, batches):
    import torch
    nx, ny, nz = shape
    t = wl.graded_film(nx, ny, nz, (nx * 5e-9, ny * 5e-9, nz * 4e-9), seed=sum(shape))
    T = mt.mt_demag_assemble_ex(mt.mt_tiles_create(mt.mt_ctx_create(0), t), prec, mt.MT_LAYOUT_DENSE)
    model = oracle.Model.from_tiles(t)
    for B in batches:
        m = np.stack([wl.m_random(t.n, seed=7 * b + 1) for b in range(B)]).astype(np.float32)
        mg = torch.tensor(m.ravel(), device="cuda")
        H = [torch.full_like(mg, float("nan")) for _ in range(2)]
        for h in H:
            mt.mt_demag_field(T, mg, h, B)
        assert torch.equal(H[0], H[1])
        Hg = H[0].cpu().numpy().reshape(B, t.n, 3)
        for b in sorted({0, B // 2, B - 1}):
            ref = np.asarray(oracle.demag_field(model, m[b].astype(np.float64))).reshape(-1, 3)
            assert np.linalg.norm(Hg[b] - ref) <= TOL[prec] * np.linalg.norm(ref), (B, b)
