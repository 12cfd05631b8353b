"""The sums over the touching tiles in every form their launch takes -- lists
shared by lanes or not, one or three blocks in flight, both states of the
operand -- with short (one layer) and long lists, against the FP64 tensor."""
import numpy as np
import pytest

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
@pytest.mark.parametrize("layout", ["dense", "stream"])
@pytest.mark.parametrize("shape,batches", [((1, 1, 1), (1, 3)), ((2, 1, 1), (1, 9)), ((7, 5, 3), (1, 4, 8, 17, 33)),
                                           ((59, 43, 1), (1, 5, 29, 64)), ((14, 13, 15), (3, 29, 64)),
                                           ((71, 69, 1), (30, 128))])
def test_near_sums(mt, ctx, prec, layout, shape, batches):
    import torch
    nx, ny, nz = shape
    t = wl.graded_film(nx, ny, nz, (nx * 5e-9, ny * 5e-9, nz * 4e-9), seed=sum(shape))
    tiles = mt.mt_tiles_create(ctx, t)
    T = mt.mt_demag_assemble_ex(tiles, prec, mt.MT_LAYOUT_DENSE if layout == "dense" else mt.MT_LAYOUT_STREAM)
    T64 = mt.mt_demag_assemble_ex(tiles, "f64", mt.MT_LAYOUT_STREAM)
    for B in batches:
        m = np.stack([wl.m_random(t.n, seed=7 * b + 1) for b in range(B)]).astype(np.float32)
        mg = torch.tensor(m.ravel(), device="cuda")
        H = torch.full_like(mg, float("nan"))
        mt.mt_demag_field(T, mg, H, B)
        Hg = H.reshape(B, -1).double()
        for b in sorted({0, B // 2, B - 1}):
            md = mg.reshape(B, -1)[b].double().contiguous()
            ref = torch.empty_like(md)
            mt.mt_demag_field_f64(T64, md, ref)
            assert float((Hg[b] - ref).norm()) <= TOL[prec] * float(ref.norm()), (B, b)
        assert bool(torch.isfinite(Hg).all())
