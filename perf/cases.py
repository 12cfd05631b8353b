"""The work this library is measured by: what programs that use it call, over
the sizes, precisions, layouts and batch widths they call it with.

Each case is one call sequence of the public binding on one tile set:

* ``field``      -- the demag product of a state (``mt_demag_field``);
* ``rhs``        -- one standalone Landau-Lifshitz right-hand side
                    (``mt_llg_rhs``);
* ``steps``      -- Runge-Kutta attempts of an integrator the program keeps,
                    from a state it loads to the state it reads back;
* ``assemble``   -- a new tensor and the first field from it, as a program
                    that varies the mesh does;
* ``threshold``  -- a thresholded copy of a kept tensor and the field from it
                    (one point of a time-against-error study).

Sizes are those of the repository's own workloads: standard problem 4 films,
standard problem 2 films, standard problem 3 cubes, graded films, prisms of
the serving stream, tetrahedral boxes.
"""
import math

import numpy as np
import torch

from paper_2107_05364_gb300 import binding as mt
from paper_2107_05364_gb300 import workloads as wl

MU0 = 4e-7 * math.pi
MS, AEX, GAMMA = 8.0e5, 1.3e-11, 2.211e5
LEX = math.sqrt(AEX / (0.5 * MU0 * MS * MS))
LAYOUTS = {"stream": mt.MT_LAYOUT_STREAM, "full": mt.MT_LAYOUT_STREAM_FULL, "dense": mt.MT_LAYOUT_DENSE}


def _case(name, op, shape, nx, ny, nz, prec="f32", layout="stream", B=1, **more):
    return dict({"name": name, "op": op, "shape": shape, "nx": nx, "ny": ny, "nz": nz, "prec": prec,
                 "layout": layout, "B": B}, **more)


def listed():
    return [
        # the smallest tensor a program asks a field of: every launch counts
        _case("field_film_400", "field", "film", 40, 10, 1),
        # one BF16 product on a mesh without any symmetry
        _case("field_graded_10800_bf16", "field", "graded", 120, 30, 3, "bf16"),
        # a caller with its own time integration asks for right-hand sides
        _case("rhs_film_2500", "rhs", "film", 100, 25, 1),
        # standard problem 4 on the coarse grid: many short steps
        _case("steps_film_400", "steps", "film", 40, 10, 1, steps=64, fixed_h=2e-13),
        # the same film at 200 x 50, the benchmark's own workload
        _case("steps_film_10000", "steps", "film", 200, 50, 1, steps=8, fixed_h=0.0),
        # standard problem 3: flower and vortex of one cube as a batch of two
        _case("steps_cube_8000_B2", "steps", "cube", 20, 20, 20, B=2, steps=8, fixed_h=0.0),
        # four states of a prism of the request stream, integrated together
        _case("steps_prism_5120_B4", "steps", "prism", 20, 16, 16, B=4, steps=8, fixed_h=0.0),
        # 64 points of a field sweep at once, FP32-like accuracy
        _case("field_film_20000_split_B64", "field", "film", 200, 50, 2, "split", "dense", B=64),
        # standard problem 2: eight film sizes on one BF16 tensor
        _case("steps_sp2_6000_bf16_B8", "steps", "sp2", 100, 20, 3, "bf16", "dense", B=8, steps=8, fixed_h=5e-14),
        # a graded mesh is new to the program: closed forms for every pair
        _case("assemble_graded_6000", "assemble", "graded", 80, 25, 3),
        # the same for tetrahedra (6 per cell)
        _case("assemble_tetra_5760", "assemble", "tetra", 12, 10, 8),
        # 40 % of the tensor's elements dropped (standard problem 4 film)
        _case("threshold_film_6400", "threshold", "film", 160, 40, 1, layout="full", fraction=0.4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dims(rng, shape, n):
    """Cells along x, y, z with about n tiles, of the shape's proportions."""
    if shape == "cube":
        s = max(2, round(n ** (1 / 3)))
        return s, s, s
    if shape == "prism":
        a = max(2, round((n / 1.5) ** (1 / 3)))
        return max(2, round(n / (a * a))), a, a
    if shape == "tetra":
        a = max(2, round((n / 6 / 1.5) ** (1 / 3)))
        return max(2, round(n / (6 * a * a))), a, max(2, a - rng.randint(0, 1))
    nz = {"film": rng.choice((1, 1, 1, 2)), "graded": rng.randint(1, 3), "sp2": 3}[shape]
    ny = max(3, round(math.sqrt(n / nz / rng.uniform(3.0, 5.0))))
    return max(4, round(n / nz / ny)), ny, nz


def _one(rng):
    op = rng.choice(("field", "field", "rhs", "steps", "steps", "batched", "batched", "assemble", "threshold"))
    if op == "field":
        shape, prec = rng.choice(("film", "graded", "cube")), rng.choice(("f32", "f32", "bf16", "split"))
        return _case("", op, shape, *_dims(rng, shape, _log_int(rng, 200, 10800)), prec, B=rng.choice((1, 1, 2, 4)))
    if op == "rhs":
        shape, prec = rng.choice(("film", "film", "graded")), rng.choice(("f32", "f32", "split"))
        return _case("", op, shape, *_dims(rng, shape, _log_int(rng, 300, 10000)), prec, B=rng.choice((1, 1, 2)))
    if op == "steps":
        shape = rng.choice(("film", "film", "cube", "prism"))
        top = {"film": 10000, "cube": 8000, "prism": 6500}[shape]
        B = rng.choice((3, 4)) if shape == "prism" else rng.choice((1, 1, 2))
        return _case("", op, shape, *_dims(rng, shape, _log_int(rng, 200, top)),
                     layout=rng.choice(("stream", "full")) if shape == "prism" else "stream", B=B,
                     steps=rng.randint(4, 8), fixed_h=0.0)
    if op == "batched":
        shape, prec = rng.choice(("film", "sp2", "cube")), rng.choice(("bf16", "split"))
        B = _log_int(rng, 5, 64)
        if rng.random() < 0.5:
            return _case("", "field", shape, *_dims(rng, shape, _log_int(rng, 1000, 18000)), prec, "dense", B=B)
        return _case("", "steps", shape, *_dims(rng, shape, _log_int(rng, 500, 6000)), prec, "dense", B=B,
                     steps=rng.randint(2, 6), fixed_h=5e-14)
    if op == "assemble":
        shape = rng.choice(("graded", "tetra"))
        return _case("", op, shape, *_dims(rng, shape, _log_int(rng, 500, 5600)))
    return _case("", "threshold", "film", *_dims(rng, "film", _log_int(rng, 1000, 6200))[:2], 1, layout="full",
                 fraction=round(rng.uniform(0.1, 0.8), 2))


def draw(rng):
    top = {k: max(work(c)[k] for c in listed()) for k in ("bytes", "flops")}
    while True:
        c = _one(rng)
        del c["name"]
        w = work(c)
        if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"]:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _tiles_count(c):
    return c["nx"] * c["ny"] * c["nz"] * (6 if c["shape"] == "tetra" else 1)


def _faces(c, seed):
    """Face coordinates along x, y, z of a cuboid tile set."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    if c["shape"] == "graded":  # 1000 x 250 x 5 nm, widths varied by up to 2 either way
        rng = np.random.default_rng([seed, 7])
        out = []
        for k, length in ((nx, 1000e-9), (ny, 250e-9), (nz, 5e-9)):
            w = 2.0 ** rng.uniform(-1.0, 1.0, k)
            f = np.concatenate([[0.0], np.cumsum(w)])
            out.append(f * (length / f[-1]))
        return out
    size = {"film": (500e-9, 125e-9, 3e-9), "sp2": (100 * LEX, 20 * LEX, 2 * LEX),
            "cube": (20 * LEX,) * 3, "prism": (nx * 4e-9, ny * 4e-9, nz * 4e-9)}[c["shape"]]
    return [np.linspace(0.0, s, k + 1) for s, k in zip(size, (nx, ny, nz))]


def _tetra_mesh(c, seed):
    """A box of cubic cells, six tetrahedra around each cell's diagonal,
    inner vertices moved by up to 5 % of a cell."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    h = 2.5e-9
    k, j, i = np.meshgrid(np.arange(nz + 1), np.arange(ny + 1), np.arange(nx + 1), indexing="ij")
    grid = np.stack([i.ravel(), j.ravel(), k.ravel()], 1).astype(np.float64)
    inner = ((grid > 0) & (grid < np.array([nx, ny, nz]))).all(1)
    grid += inner[:, None] * np.random.default_rng([seed, 11]).uniform(-0.05, 0.05, grid.shape)
    at = lambda i, j, k: i + (nx + 1) * (j + (ny + 1) * k)
    k, j, i = (a.ravel() for a in np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"))
    tets = []
    for order in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        p = [i, j, k]
        v = [at(*p)]
        for a in order:
            p = [q + (b == a) for b, q in enumerate(p)]
            v.append(at(*p))
        tets.append(np.stack(v, 1))
    return grid * h, np.stack(tets, 1).reshape(-1, 4).astype(np.int32)


def _state(c, seed):
    """B unit vector fields, FP32: a smooth texture about a direction of its
    own per simulation, with a little noise, as a run meets it."""
    n, B = _tiles_count(c), c["B"]
    rng = np.random.default_rng([seed, 3])
    d = rng.normal(size=(B, 1, 3))
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    s = np.arange(n)[None, :, None] / n
    wave = 0.6 * np.sin(2 * np.pi * (rng.uniform(0.5, 3.0, (B, 1, 3)) * s + rng.uniform(size=(B, 1, 3))))
    m = d + wave + 0.05 * rng.uniform(-1.0, 1.0, (B, n, 3))
    return (m / np.linalg.norm(m, axis=-1, keepdims=True)).astype(np.float32)


def _params(c):
    """alpha (B,) and applied fields (B, 3) in A/m: points of a field sweep."""
    B = c["B"]
    t = np.linspace(1.0, -1.0, B) if B > 1 else np.ones(1)
    Ha = (np.stack([-24.6e-3 * t, 4.3e-3 * np.ones(B), 2.0e-3 * t], 1)) / MU0
    return np.array([(0.02, 0.1, 0.5)[b % 3] for b in range(B)]), Ha


def _ku(c):
    return 0.1 * 0.5 * MU0 * MS * MS if c["shape"] == "cube" else 0.0


def _opts(c):
    return mt.ode_opts(rtol=1e-5, atol=1e-5, h0=1e-14, hmax=1e-11, fixed_h=c["fixed_h"])


_CTX = []


def _ctx():
    """The program's one library context."""
    if not _CTX:
        _CTX.append(mt.mt_ctx_create(torch.cuda.current_device()))
    return _CTX[0]


def prepare(case, seed):
    c = case
    n, B = _tiles_count(c), c["B"]
    if c["shape"] == "tetra":
        tiles = mt.mt_tiles_create_tetra(_ctx(), *_tetra_mesh(c, seed), MS, AEX, 0.0)
    else:
        tiles = mt.mt_tiles_create(_ctx(), wl.grid_tiles(*_faces(c, seed), MS, AEX, _ku(c)))
    m = torch.from_numpy(_state(c, seed)).cuda()
    s = {"case": c, "tiles": tiles, "m": m, "H": torch.empty_like(m)}
    if c["op"] != "assemble":
        s["T"] = mt.mt_demag_assemble_ex(tiles, c["prec"], LAYOUTS[c["layout"]])
    if c["op"] in ("rhs", "steps"):
        alpha, Ha = _params(c)
        s["params"], s["keep"] = mt.llg_params(B, alpha=alpha, Ha=Ha)
        s["tau"] = torch.empty(B, device="cuda")
    if c["op"] == "steps":
        s["I"] = mt.mt_integrator_create(s["T"], s["params"], _opts(c), B)
    return s


def run(state):
    c, B = state["case"], state["case"]["B"]
    m, H = state["m"], state["H"]
    if c["op"] == "field":
        mt.mt_demag_field(state["T"], m, H, B)
        return H
    if c["op"] == "rhs":
        mt.mt_llg_rhs(state["T"], state["params"], m, H, state["tau"], B)
        return H, state["tau"]
    if c["op"] == "steps":
        I = state["I"]
        I.set_state(m)
        I.step(c["steps"])
        return I.get_state(H)
    if c["op"] == "assemble":
        T = mt.mt_demag_assemble(state["tiles"], c["prec"])
        mt.mt_demag_field(T, m, H, B)
        T.close()
        return H
    T, cut, kept = mt.mt_tensor_threshold(state["T"], c["fraction"])
    mt.mt_demag_field(T, m, H, B)
    T.close()
    return H, cut, kept


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Tensor bytes: each 3x3 block of two tiles is symmetric with trace 0, so
    5 values (3 for a single layer, whose xz and yz vanish), and for tiles of
    one shape block (i, j) is block (j, i).  Flops of a product: 2 per matrix
    element that can differ from zero and simulation."""
    c = case
    n, B = _tiles_count(c), c["B"]
    flat = c["shape"] != "tetra" and c["nz"] == 1
    blocks = n * n if c["shape"] in ("graded", "tetra") else n * (n + 1) // 2
    tensor = blocks * (3 if flat else 5) * (2 if c["prec"] == "bf16" else 4)
    product = (10 if flat else 18) * n * n * B
    vec = 12 * n * B
    if c["op"] == "field":
        return {"bytes": tensor + 2 * vec, "flops": product}
    if c["op"] == "rhs":
        return {"bytes": tensor + 2 * vec, "flops": product + 60 * n * B}
    if c["op"] == "steps":
        rhs = 1 + 6 * c["steps"]
        return {"bytes": rhs * (tensor + 2 * vec) + 2 * vec, "flops": rhs * (product + 90 * n * B)}
    if c["op"] == "assemble":
        # per block: 8 distances, 3 logarithms, 6 angles (tetrahedron: 4
        # distances, 6 logarithms, 4 angles), about 20 operations each
        return {"bytes": 2 * tensor + 2 * vec, "flops": product + 450 * blocks}
    kept = 1.0 - c["fraction"]
    return {"bytes": int(n * n * 16 * (1 + 2 * kept)) + 2 * vec, "flops": int(product * kept)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the closed forms
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _cuboid(r, e):
    """The six entries of the tensor of cuboids with full edges e at the
    offsets r (each a triple of arrays), H = -N M."""
    d = [[r[a] - s * 0.5 * e[a] for s in (-1.0, 1.0)] for a in range(3)]
    out = [0.0] * 6
    for q in range(8):
        f = (q & 1, q >> 1 & 1, q >> 2 & 1)
        x, y, z = (d[a][f[a]] for a in range(3))
        s = 1.0 if sum(f) % 2 else -1.0
        R = torch.sqrt(x * x + y * y + z * z)

        def angle(u, v, w):
            return torch.where(w == 0, torch.zeros_like(R), torch.atan(u * v / torch.where(w == 0, R, w * R)))

        def log(w, u, v):  # log(w + R), from (u^2 + v^2) / (R - w) where w < 0
            return torch.where(w < 0, torch.log(u * u + v * v) - torch.log(R + w.abs()), torch.log(R + w.abs()))

        for k, v in ((0, -s * angle(y, z, x)), (3, -s * angle(x, z, y)), (5, -s * angle(x, y, z)),
                     (1, s * log(z, x, y)), (2, s * log(y, x, z)), (4, s * log(x, y, z))):
            out[k] = out[k] + v
    return [v / (4 * math.pi) for v in out]


def _tetra_entries(r, V):
    """The same for tetrahedra V (n, 4, 3) at the points r (k, 1, 3)."""
    N = [0.0] * 6
    R = [V[None, :, a] - r for a in range(4)]
    L = [x.norm(dim=-1) for x in R]
    for f in range(4):
        a, b, c = [q for q in range(4) if q != f]
        nf = torch.linalg.cross(V[:, b] - V[:, a], V[:, c] - V[:, a])
        flip = ((nf * (V[:, f] - V[:, a])).sum(-1) > 0).to(V.dtype)
        nf = nf * (1 - 2 * flip)[:, None]
        nf = nf / nf.norm(dim=-1, keepdim=True)
        sign = 1 - 2 * flip
        triple = (R[a] * torch.linalg.cross(R[b], R[c])).sum(-1) * sign
        dot = lambda p, q: (R[p] * R[q]).sum(-1)
        omega = -2 * torch.atan2(triple, L[a] * L[b] * L[c] + dot(a, b) * L[c] + dot(a, c) * L[b] + dot(b, c) * L[a])
        g = -omega[..., None] * nf
        for p, q in ((a, b), (b, c), (c, a)):
            t = V[:, q] - V[:, p]
            t = t / t.norm(dim=-1, keepdim=True)
            u = torch.linalg.cross(t, nf) * sign[:, None]
            sp, sq = (R[p] * t).sum(-1), (R[q] * t).sum(-1)
            li = torch.where(sp + sq >= 0, torch.log((L[q] + sq) / (L[p] + sp)), torch.log((L[p] - sp) / (L[q] - sq)))
            g = g - li[..., None] * u
        for k, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
            N[k] = N[k] + 0.5 * (g[..., i] * nf[:, j] + g[..., j] * nf[:, i])
    return [v / (4 * math.pi) for v in N]


def _demag(c, seed):
    """x (B, n, 3) -> H = -N x in 64 bits."""
    dev = _device()
    n = _tiles_count(c)
    pairs = ((0, 0, 0), (0, 1, 1), (0, 2, 2), (1, 0, 1), (1, 1, 3), (1, 2, 4), (2, 0, 2), (2, 1, 4), (2, 2, 5))
    if c["shape"] in ("graded", "tetra"):
        if c["shape"] == "tetra":
            verts, tets = _tetra_mesh(c, seed)
            V = torch.tensor(verts[tets] / 2.5e-9, dtype=torch.float64, device=dev)
            C = V.mean(1)
            block = lambda i: _tetra_entries(C[i, None], V)
        else:
            F = [f / 1e-9 for f in _faces(c, seed)]
            C, E = (torch.tensor(np.stack([a.ravel() for a in np.meshgrid(*v[::-1], indexing="ij")][::-1], 1),
                                 device=dev) for v in ([0.5 * (f[1:] + f[:-1]) for f in F], [np.diff(f) for f in F]))
            block = lambda i: _cuboid([C[i, None, a] - C[None, :, a] for a in range(3)], [E[None, :, a] for a in range(3)])

        def apply(x):
            H = torch.zeros_like(x)
            step = max(1, (1 << 22) // n)
            for i0 in range(0, n, step):
                N = block(slice(i0, min(n, i0 + step)))
                for a, b, k in pairs:
                    H[:, i0:i0 + step, a] -= x[:, :, b] @ N[k].T
            return H
        return apply
    # one shape: the product is a convolution over the lattice offsets
    dims = (c["nx"], c["ny"], c["nz"])
    e = [(f[1] - f[0]) for f in _faces(c, seed)]
    off = torch.meshgrid(*[torch.tensor((np.fft.fftfreq(2 * k) * 2 * k) * (q / e[2]), device=dev)
                           for k, q in zip(dims, e)][::-1], indexing="ij")
    N = _cuboid(off[::-1], [torch.full_like(off[0], q / e[2]) for q in e])
    K = [torch.fft.rfftn(v) for v in N]
    full = [2 * k for k in dims[::-1]]

    def apply(x):
        H = torch.empty_like(x)
        for b0 in range(0, x.shape[0], 8):
            xb = x[b0:b0 + 8].reshape(-1, *dims[::-1], 3)
            X = [torch.fft.rfftn(xb[..., a], s=full, dim=(1, 2, 3)) for a in range(3)]
            for a in range(3):
                Y = sum(K[k] * X[b] for p, b, k in pairs if p == a)
                y = torch.fft.irfftn(Y, s=full, dim=(1, 2, 3))[:, :dims[2], :dims[1], :dims[0]]
                H[b0:b0 + 8, :, a] = -y.reshape(xb.shape[0], n)
        return H
    return apply


def _thresholded(c, seed, x):
    """H of the single-layer tensor without the smallest elements."""
    dev = x.device
    F = _faces(c, seed)
    C, E = (np.stack([a.ravel() for a in np.meshgrid(*v[::-1], indexing="ij")][::-1], 1) / 1e-9
            for v in ([0.5 * (f[1:] + f[:-1]) for f in F], [np.diff(f) for f in F]))
    C, E = torch.tensor(C, device=dev), torch.tensor(E[0], device=dev)
    n = C.shape[0]
    P = torch.empty(4, n, n, dtype=torch.float32, device=dev)
    for i0 in range(0, n, 512):
        N = _cuboid([C[i0:i0 + 512, None, a] - C[None, :, a] for a in range(3)], [E[a] for a in range(3)])
        for p, k in enumerate((0, 1, 3, 5)):
            P[p, i0:i0 + 512] = N[k].float()
    mag = torch.cat([P.abs().flatten(), P[1].abs().flatten()])
    mag = mag[mag > 0].sort().values
    k = int(c["fraction"] * mag.numel())
    cut = mag[k] if k else torch.zeros((), device=dev)
    del mag
    H = torch.zeros_like(x)
    for a, b, p in ((0, 0, 0), (0, 1, 1), (1, 0, 1), (1, 1, 2), (2, 2, 3)):
        for i0 in range(0, n, 512):
            v = P[p, i0:i0 + 512]
            H[:, i0:i0 + 512, a] -= x[:, :, b] @ torch.where(v.abs() >= cut, v, torch.zeros_like(v)).double().T
    return H


def _field_of(c, seed):
    """m (B, n, 3) -> effective field without the demag part, 64 bits."""
    dev = _device()
    n, B = _tiles_count(c), c["B"]
    F = _faces(c, seed)
    dims = (c["nx"], c["ny"], c["nz"])
    Ha = torch.tensor(_params(c)[1], device=dev)[:, None, :]
    ka = 2 * _ku(c) / (MU0 * MS)

    def local(m):
        v = m.reshape(B, *dims[::-1], 3)
        H = torch.zeros_like(v)
        for a in range(3):
            ax = 3 - a  # x runs fastest
            if dims[a] < 2:
                continue
            h = torch.tensor(np.diff(F[a]), device=dev)
            mid = torch.tensor(0.5 * (F[a][1:] + F[a][:-1]), device=dev)
            shape = [1] * 5
            shape[ax] = -1
            d = v.narrow(ax, 1, dims[a] - 1) - v.narrow(ax, 0, dims[a] - 1)
            gap = (mid[1:] - mid[:-1])
            k = 2 * AEX / (MU0 * MS)
            H.narrow(ax, 0, dims[a] - 1).add_(d * (k / (h[:-1] * gap)).reshape(shape))
            H.narrow(ax, 1, dims[a] - 1).sub_(d * (k / (h[1:] * gap)).reshape(shape))
        H = H.reshape(B, n, 3) + Ha
        if ka:
            H[..., 2] += ka * m[..., 2]
        return H
    return local


_A = ((), (1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
      (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
      (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
      (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
_E = (71 / 57600, 0.0, -71 / 16695, 71 / 1920, -17253 / 339200, 22 / 525, -1 / 40)


def exact(case, seed):
    c = case
    dev = _device()
    B = c["B"]
    m = torch.tensor(_state(c, seed), dtype=torch.float64, device=dev)
    if c["op"] == "threshold":
        return _thresholded(c, seed, MS * m), None, None
    demag = _demag(c, seed)
    if c["op"] in ("field", "assemble"):
        return demag(MS * m)
    local = _field_of(c, seed)
    alpha = torch.tensor(_params(c)[0], device=dev)[:, None, None]
    g1 = GAMMA / (1 + alpha * alpha)
    torque = [None]

    def f(m):
        a = torch.linalg.cross(m, demag(MS * m) + local(m))
        torque[0] = a.norm(dim=-1).amax(-1) / MS
        return -g1 * (a + alpha * torch.linalg.cross(m, a))

    if c["op"] == "rhs":
        k = f(m)
        return k, torque[0]
    if _tiles_count(c) > 3000 and c["shape"] in ("graded", "tetra"):
        return None
    fixed = c["fixed_h"]
    h = torch.full((B, 1, 1), fixed or 1e-14, dtype=torch.float64, device=dev)
    k1 = f(m)
    for _ in range(c["steps"]):
        hs = h if fixed else h.clamp(max=1e-11)
        k = [k1]
        for s in range(1, 7):
            y = m + hs * sum(a * q for a, q in zip(_A[s], k))
            k.append(f(y))
        e = hs * sum(w * q for w, q in zip(_E, k))
        err = (e / (1e-5 + 1e-5 * torch.maximum(m.abs(), y.abs()))).square().mean((1, 2), keepdim=True).sqrt()
        take = torch.ones_like(err, dtype=torch.bool) if fixed else err <= 1.0
        m = torch.where(take, y / y.norm(dim=-1, keepdim=True), m)
        k1 = torch.where(take, k[6], k1)
        if not fixed:
            h = (hs * (0.9 * err.clamp(min=1e-30) ** -0.2).clamp(0.2, 5.0)).clamp(max=1e-11)
    return m
