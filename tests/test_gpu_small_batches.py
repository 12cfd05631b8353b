"""The one-kernel integrator with several simulations (grouped between CTA
barriers, their polls side by side): each simulation does what it does alone,
to the bit, also beside finished ones; the group widths and poll widths change
over these sizes.  And a batch does not cost as much as its simulations one
after the other."""
import time

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


def _setup(mt, ctx, shape, B):
    nx, ny, nz = shape
    t = wl.film(nx, ny, nz, size=(nx * 6e-9, ny * 6e-9, nz * 4e-9))
    T = mt.mt_demag_assemble(mt.mt_tiles_create(ctx, t), "f32")
    alpha = np.array([(0.9, 0.1, 0.5, 0.02)[b % 4] for b in range(B)])
    Ha = np.stack([np.linspace(4e5, -4e5, B), np.full(B, 3e5), np.linspace(0, 2e5, B)], 1)
    m0 = np.stack([wl.m_noisy(t.n, (1, 0.5, 0.2 + b), 0.3, seed=b) for b in range(B)]).astype(np.float32)
    return t, T, alpha, Ha, m0


def _integrator(mt, T, alpha, Ha, m0):
    p, keep = mt.llg_params(len(alpha), alpha=alpha, Ha=Ha)
    I = mt.Integrator(T, p, mt.ode_opts(rtol=1e-5, atol=1e-5), len(alpha))
    assert I.path() == mt.MT_PATH_PERSISTENT
    I.set_state(m0.ravel())
    return I


@pytest.mark.parametrize("shape,B", [((1, 1, 1), 3), ((1, 1, 1), 5), ((2, 1, 1), 128), ((10, 1, 1), 4),
                                     ((5, 3, 1), 17), ((16, 8, 1), 7), ((19, 8, 1), 4), ((32, 8, 2), 3),
                                     ((19, 9, 3), 3), ((19, 9, 3), 6), ((40, 25, 1), 4), ((30, 10, 2), 16)])
def test_each_simulation_as_alone(mt, ctx, shape, B):
    t, T, alpha, Ha, m0 = _setup(mt, ctx, shape, B)
    I = _integrator(mt, T, alpha, Ha, m0)
    I.step(3)
    st, stats = I.relax(0.2, 3e-11, check=False)  # some finish long before others
    got = I.get_state()
    if t.n > 1 and B > 3:
        assert len({s["n_accept"] for s in stats}) > 1
    for b in sorted({0, 1, B // 2, B - 1}):
        J = _integrator(mt, T, alpha[b:b + 1], Ha[b:b + 1], m0[b])
        J.step(3)
        _, s1 = J.relax(0.2, 3e-11, check=False)
        assert s1[0] == stats[b], b
        assert np.array_equal(J.get_state()[0], got[b]), b


def test_a_batch_costs_less_than_its_simulations(mt, ctx):
    # eight warps own sixteen simulations two each, and everything else of a
    # stage is a few hundred cycles per simulation: an attempt of sixteen takes
    # two to four attempts' time of one (one after the other: nine)
    def attempt(B):
        t, T, alpha, Ha, m0 = _setup(mt, ctx, (10, 1, 1), B)
        p, keep = mt.llg_params(B, alpha=alpha, Ha=Ha)
        I = mt.Integrator(T, p, mt.ode_opts(fixed_h=1e-15), B)
        I.set_state(m0.ravel())
        I.step(64)
        best = 1e9
        for _ in range(7):
            t0 = time.perf_counter()
            I.step(256)
            I.get_state()
            best = min(best, time.perf_counter() - t0)
        return best

    assert attempt(16) < 6 * attempt(1)
