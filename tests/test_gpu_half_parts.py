"""The half-stored product where its CTAs' ranges split groups and super-rows
in every way: one unit per CTA (fewer units than SMs), several CTAs inside one
group, ranges over many short super-rows, one ragged panel; one, two and four
simulations per read and partly filled groups of them.  Against the FP64 oracle
and, for finished simulations, against the untouched rest of the field."""
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


@pytest.mark.parametrize("shape", [(1, 1, 1), (17, 1, 1), (16, 8, 1), (43, 3, 1), (10, 10, 4), (37, 23, 1),
                                   (12, 11, 13), (90, 33, 1)])
def test_field_matches_oracle(mt, ctx, shape):
    import torch
    nx, ny, nz = shape
    t = wl.film(nx, ny, nz, size=(nx * 5e-9, ny * 5e-9, nz * 4e-9))
    T = mt.mt_demag_assemble_ex(mt.mt_tiles_create(ctx, t), "f32", mt.MT_LAYOUT_STREAM_HALF)
    model = oracle.Model.from_tiles(t)
    for B in (1, 2, 3, 4, 7):
        m = np.stack([wl.m_random(t.n, seed=5 * b + 2) for b in range(B)]).astype(np.float32)
        mg = torch.tensor(m.ravel(), device="cuda")
        H = torch.full_like(mg, float("nan"))
        for _ in range(2):
            mt.mt_demag_field(T, mg, H, B)
        Hg = H.cpu().numpy().reshape(B, t.n, 3)
        for b in sorted({0, B - 1}):
            ref = np.asarray(oracle.demag_field(model, m[b].astype(np.float64))).reshape(-1, 3)
            # FP32 storage and sums: the precision's stated field error
            assert np.linalg.norm(Hg[b] - ref) <= 1e-6 * np.linalg.norm(ref), (B, b)


def test_finished_simulations_leave_the_rest_alone(mt, ctx):
    # four simulations, the first already at its end time: the group of four
    # still serves the others, as each alone
    t = wl.film(60, 20, 1, size=(300e-9, 100e-9, 3e-9))
    T = mt.mt_demag_assemble_ex(mt.mt_tiles_create(ctx, t), "f32", mt.MT_LAYOUT_STREAM_HALF)
    alpha = np.array([1.0, 0.5, 0.1, 0.02])
    m0 = np.stack([np.tile([[1.0, 0.0, 0.0]], (t.n, 1))] +
                  [wl.m_noisy(t.n, (1, 1, 1), 0.2, seed=b) for b in (1, 2, 3)]).astype(np.float32)
    p, keep = mt.llg_params(4, alpha=alpha, Ha=(2e6, 0.0, 0.0))  # the first one is at rest in this field
    I = mt.Integrator(T, p, mt.ode_opts(rtol=1e-5, atol=1e-5), 4)
    I.set_state(m0.ravel())
    st, stats = I.relax(0.3, 2e-12, check=False)
    assert stats[0]["n_accept"] < min(s["n_accept"] for s in stats[1:])
    got = I.get_state()
    for b in (1, 3):
        p1, k1 = mt.llg_params(1, alpha=alpha[b], Ha=(2e6, 0.0, 0.0))
        J = mt.Integrator(T, p1, mt.ode_opts(rtol=1e-5, atol=1e-5), 1)
        J.set_state(m0[b].ravel())
        _, s1 = J.relax(0.3, 2e-12, check=False)
        # sums in another order: FP32 round-off grown over the steps of 2 ps
        assert abs(s1[0]["t"] - stats[b]["t"]) <= 1e-3 * s1[0]["t"]
        assert np.abs(J.get_state()[0] - got[b]).max() < 1e-3
