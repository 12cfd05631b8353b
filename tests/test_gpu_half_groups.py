"""Half-stored tensors with four and more simulations to a read while some of a
group have finished or have not begun: fixed steps, so that the bound is set by
rounding, against the FP64 oracle and the full storage; and the request server
with four and five slots, jobs entering and leaving at different times, against
the same jobs one by one."""
import numpy as np
import pytest

import oracle
from paper_2107_05364_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
MU0 = 4e-7 * np.pi


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


@pytest.mark.parametrize("B,at_rest", [(4, (0,)), (4, (1, 2, 3)), (5, (4,)), (6, (0, 1, 2, 3)), (8, (2, 5, 7))])
def test_fixed_steps_beside_finished_simulations(mt, ctx, B, at_rest):
    # simulations at rest finish before their first step; the others take 8
    nx, ny = 60, 20
    t = wl.film(nx, ny, 1, size=(nx * 5e-9, ny * 5e-9, 3e-9))
    Ha, h = (2e6, 0.0, 0.0), 1e-13
    m0 = np.stack([np.tile([[1.0, 0.0, 0.0]], (t.n, 1)) if b in at_rest else wl.m_noisy(t.n, (1, 1, 1), 0.2, seed=b)
                   for b in range(B)]).astype(np.float32)
    tiles = mt.mt_tiles_create(ctx, t)
    p, keep = mt.llg_params(B, alpha=0.05, Ha=Ha)
    out = {}
    for layout in (mt.MT_LAYOUT_STREAM_HALF, mt.MT_LAYOUT_STREAM_FULL):
        I = mt.Integrator(mt.mt_demag_assemble_ex(tiles, "f32", layout), p, mt.ode_opts(fixed_h=h), B)
        I.set_path(mt.MT_PATH_GRAPH)
        I.set_state(m0.ravel())
        st, stats = I.relax(0.3, 8 * h, check=False)
        # (a ninth step may close the round-off of the summed time)
        assert all(abs(s["t"] - (0 if b in at_rest else 8 * h)) <= 1e-6 * h for b, s in enumerate(stats))
        out[layout] = I.get_state().copy()
    half = out[mt.MT_LAYOUT_STREAM_HALF]
    # 8 steps of rounded fields: the bound of the half storage's step test
    assert np.abs(half - out[mt.MT_LAYOUT_STREAM_FULL]).max() <= 3e-6
    model = oracle.Model.from_tiles(t)
    for b in range(B):
        if b in at_rest:
            assert np.abs(half[b] - m0[b]).max() <= 1e-6
            continue
        so, mo, _, _ = oracle.integrate(model, m0[b].astype(np.float64), oracle.llg_params(alpha=0.05, Ha=Ha),
                                        oracle.ode_opts(fixed_h=h), 0.0, 8 * h, 1)
        assert so == oracle.OK
        assert np.abs(half[b] - mo).max() <= 3e-6, b


@pytest.mark.parametrize("slots", [4, 5])
def test_server_slots_come_and_go(mt, ctx, slots):
    # relaxed to a torque of 1e-5 with the integrator's error below it, so that
    # the stopping points agree to 1e-4 (as between the storages)
    t = wl.film(70, 40, 1, size=(350e-9, 200e-9, 3e-9))
    jobs = [dict(m0=wl.m_noisy(t.n, (np.cos(k), np.sin(k), 0.3), 0.3, seed=k), alpha=(0.9, 0.5, 0.3)[k % 3],
                 Ha=(30e-3 + 8e-3 * k) / MU0 * np.array([np.cos(1.3 * k), np.sin(1.3 * k), 0.1])) for k in range(7)]

    def run(which, max_batch):
        S = mt.Server(ctx, max_batch=max_batch, layout=mt.MT_LAYOUT_STREAM_HALF, opts=mt.ode_opts(rtol=1e-7, atol=1e-7))
        g = S.add_geometry(t)
        ids = [S.submit(g, j["m0"], alpha=j["alpha"], Ha=j["Ha"], tol=1e-5, t_max=20e-9) for j in which]
        out = [S.wait(i, 120.0, geometry=g) for i in ids]
        S.close()
        return out

    mix = run(jobs, slots)
    ends = [r["t_done"] for _, r, _ in mix]
    assert len(set(ends)) > 1
    for k, (s, r, m) in enumerate(mix):
        s1, r1, m1 = run([jobs[k]], 1)[0]
        assert s == 0 and s1 == 0 and r["status"] == 0 and r1["status"] == 0
        assert np.abs(m - m1).max() <= 1e-4, k
