"""What a server charges an engine against its budget is what the engine takes
on the device: dense tensors with many slots, whose partial sums outweigh a
small tensor, half-stored tensors and their column work area, full ones.  Each
in a process of its own: the driver keeps small blocks of engines that are
gone, and the next engine would seem to take less."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# about 15 allocations of an engine may each be rounded up by 2 MB (and the
# kernels' code is loaded); 4 MB of the charge stand for small ones
ROUNDING = 15 * 2 << 20
FLAT = 4 << 20

CHILD = """
import json, sys
import numpy as np, torch
from paper_2107_05364_gb300 import binding as mt, workloads as wl

def solid(nx, ny, nz):
    return wl.grid_tiles(np.linspace(0, nx * 5e-9, nx + 1), np.linspace(0, ny * 5e-9, ny + 1),
                         np.linspace(0, nz * 5e-9, nz + 1), 8e5, 1.3e-11, 0.0)

t = eval(sys.argv[1])
ctx = mt.mt_ctx_create(0)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
S = mt.Server(ctx, opts=mt.ode_opts(rtol=1e-5, atol=1e-5), **json.loads(sys.argv[2]))
g = S.add_geometry(t)
s, r, _ = S.wait(S.submit(g, wl.m_noisy(t.n), alpha=0.5, tol=1e-1, t_max=1e-14), 60.0)
assert s == 0
st = S.stats()
print(json.dumps([st["bytes_in_use"], before - torch.cuda.mem_get_info()[0], st["budget"]]))
S.close()
"""


@pytest.mark.parametrize("tiles,opts", [
    ("wl.film(50, 10, 1)", dict(max_batch=128, prec="split", layout="MT_LAYOUT_DENSE")),
    ("wl.film(80, 52, 1)", dict(max_batch=4)),
    ("solid(16, 16, 12)", dict(max_batch=2, prec="bf16")),
    ("solid(18, 25, 10)", dict(max_batch=8)),
    ("wl.graded_film(60, 50, 1, (300e-9, 200e-9, 3e-9), seed=4)", dict(max_batch=64)),
    # 18.0 MB without the blocks kept apart, 20.2 with them: does not fit 19.5
    ("solid(10, 10, 10)", dict(max_batch=1, prec="bf16", hbm_budget_bytes=19500000)),
])
def test_charge_is_what_an_engine_takes(tiles, opts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2107_05364_gb300 import binding, build
    build.build()
    if "layout" in opts:
        opts = dict(opts, layout=getattr(binding, opts["layout"]))
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", CHILD, tiles, json.dumps(opts)], cwd=root, capture_output=True, text=True,
                         timeout=120)
    assert out.returncode == 0, out.stderr[-2000:]
    charged, taken, budget = json.loads(out.stdout.strip().splitlines()[-1])
    assert charged <= budget
    assert taken - ROUNDING <= charged <= taken + FLAT, (charged, taken)
