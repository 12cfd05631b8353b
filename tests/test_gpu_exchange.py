"""The one-kernel integrator's exchange between CTAs, at the sizes where its
splits change: one tile per CTA and fewer tiles than SMs, one row more than
the SMs, several polls per thread, rows read from L2, multi-layer (6-plane)
rows, and more simulations than warps (a warp then owns several).  The first
step is far too long, so attempts are rejected and the stage-2 input comes
from the published state.  Against the graph path: the same equation, control
and counters, row sums in another order."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("shape,B", [((1, 1, 1), 1), ((2, 1, 1), 1), ((5, 3, 1), 9), ((17, 9, 1), 2), ((19, 8, 2), 1),
                                     ((32, 16, 2), 1), ((40, 26, 1), 1), ((60, 30, 1), 2),
                                     ((60, 30, 1), 1), ((14, 12, 12), 3), ((40, 20, 2), 9)])
def test_rejections_and_splits_match_graph(mt, ctx, shape, B):
    nx, ny, nz = shape
    t = wl.film(nx, ny, nz, size=(nx * 6e-9, ny * 6e-9, nz * 4e-9))
    T = mt.mt_demag_assemble(mt.mt_tiles_create(ctx, t), "f32")
    Ha = np.stack([np.linspace(4e4, -4e4, B), np.full(B, 3e4), np.linspace(0, 2e4, B)], 1)
    p, keep = mt.llg_params(B, alpha=[(0.02, 0.1, 0.5)[b % 3] for b in range(B)], Ha=Ha)
    m0 = np.stack([wl.m_noisy(t.n, (1, 0.5, 0.2 + b), 0.3, seed=b) for b in range(B)]).astype(np.float32)
    got = {}
    for path in (mt.MT_PATH_PERSISTENT, mt.MT_PATH_GRAPH):
        I = mt.Integrator(T, p, mt.ode_opts(rtol=1e-5, atol=1e-5, h0=2e-12, hmax=2e-12), B)
        I.set_path(path)
        I.set_state(m0.ravel())
        I.step(7)
        I.step(5)  # a second launch starts from global memory again
        got[path] = I.get_state(), I.stats()
    a, sa = got[mt.MT_PATH_PERSISTENT]
    b, sb = got[mt.MT_PATH_GRAPH]
    for x, y in zip(sa, sb):
        assert (x["n_accept"], x["n_reject"], x["n_rhs"]) == (y["n_accept"], y["n_reject"], y["n_rhs"])
    if t.n > 2:  # (one tile barely moves: its first step may pass)
        assert all(x["n_reject"] > 0 for x in sa)
    # 73 right-hand sides, each field rounded at 1e-7 of itself, over steps of
    # up to a radian of precession
    assert np.abs(a - b).max() < 1e-5
