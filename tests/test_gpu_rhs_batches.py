"""The standalone right-hand side beyond the simulations whose parameters one
launch carries (64): every simulation of a batch against a call of its own."""
import numpy as np
import pytest

from paper_2107_05364_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
# two FP32 fields, each within 3e-7 of the exact one, through a right-hand side
# that is linear in the field: 6e-7, and a few roundings of 6e-8
TOL = 1e-6


@pytest.fixture(scope="module")
def mt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2107_05364_gb300 import build
    build.build()
    from paper_2107_05364_gb300 import binding
    return binding


@pytest.mark.parametrize("B", [1, 64, 65, 130])
def test_batch_matches_single_calls(mt, B):
    import torch
    t = wl.graded_film(23, 7, 2, (200e-9, 80e-9, 6e-9), seed=3)
    T = mt.mt_demag_assemble(mt.mt_tiles_create(mt.mt_ctx_create(0), t), "f32")
    alphas = [0.02 + 0.01 * b for b in range(B)]
    Ha = np.array([[1e4 * (b + 1), -3e3 * b, 5e3] for b in range(B)])
    m = np.stack([wl.m_random(t.n, seed=5 * b) for b in range(B)]).astype(np.float32)
    mg = torch.tensor(m, device="cuda").reshape(B, -1)
    p, keep = mt.llg_params(B, alpha=alphas, Ha=Ha)
    k, tau = torch.full_like(mg, float("nan")), torch.full((B,), 9.0, device="cuda")
    mt.mt_llg_rhs(T, p, mg.reshape(-1), k.reshape(-1), tau, B=B)
    for b in sorted({0, B // 2, 63 % B, 64 % B, B - 1}):
        p1, keep1 = mt.llg_params(1, alpha=alphas[b], Ha=Ha[b])
        k1, tau1 = torch.empty_like(mg[b]), torch.empty(1, device="cuda")
        mt.mt_llg_rhs(T, p1, mg[b].contiguous(), k1, tau1)
        assert float((k[b] - k1).norm()) <= TOL * float(k1.norm()), b
        assert abs(float(tau[b]) - float(tau1)) <= 2 * TOL * float(tau1), b
    assert bool(torch.isfinite(k).all())
