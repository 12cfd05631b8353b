"""Several integrators of the one-kernel path alive at once: a later one that
needs less shared memory leaves the earlier ones as they were."""
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


@pytest.mark.parametrize("shapes,B", [(((31, 5, 1), (10, 3, 1)), 1), (((50, 22, 1), (40, 20, 1)), 1),
                                      (((30, 10, 2), (8, 5, 4)), 2), (((15, 10, 1), (2, 1, 1)), 6),
                                      (((50, 40, 1), (46, 36, 1)), 1)])
def test_the_earlier_integrator_still_steps(mt, shapes, B):
    ctx = mt.mt_ctx_create(0)
    p, keep = mt.llg_params(B, alpha=0.1, Ha=(1e4, -2e4, 5e3))
    made = []
    for nx, ny, nz in shapes:
        t = wl.film(nx, ny, nz, size=(nx * 5e-9, ny * 5e-9, nz * 3e-9))
        T = mt.mt_demag_assemble(mt.mt_tiles_create(ctx, t), "f32")
        I = mt.Integrator(T, p, mt.ode_opts(fixed_h=1e-14), B)
        assert I.path() == mt.MT_PATH_PERSISTENT
        m0 = np.stack([wl.m_noisy(t.n, seed=b) for b in range(B)]).astype(np.float32)
        I.set_state(m0.ravel())
        if not made:
            I.step(5)
            alone = I.get_state().copy()
            I.set_state(m0.ravel())
        made.append(I)
    for I in made:
        I.step(5)
    assert np.array_equal(made[0].get_state(), alone)
