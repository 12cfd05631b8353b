"""The closed forms of assembly on both sides of their switches (series or
full function of the combined arguments; shared tetrahedron edges), against
the oracle: self and touching tiles, tiles in one another's face planes, and
distant tiles, in metres and in units where products of lengths would leave
the FP64 range."""
import types

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


@pytest.mark.parametrize("unit", [1.0, 1e-31, 1e28])
@pytest.mark.parametrize("layers", [1, 3])
def test_cuboid_blocks(mt, ctx, unit, layers):
    g = wl.graded_film(37, 3, layers, (185e-9, 15e-9, 4e-9 * layers), seed=5)
    t = types.SimpleNamespace(centre=g.centre * unit, edge=g.edge * unit, Ms=g.Ms, Aex=g.Aex, Ku=g.Ku, axis=g.axis,
                              nbr=None)
    n = g.n
    pairs = np.stack(np.meshgrid(np.arange(n), np.arange(n), indexing="ij"), -1).reshape(-1, 2)
    got = mt.mt_demag_blocks(mt.mt_tiles_create(ctx, t), pairs).reshape(n, n, 6)
    # in metres the oracle's own forms hold; the tensor has no unit
    ref = oracle.demag_blocks(g.centre, g.edge, pairs).reshape(n, n, 6)
    # an entry sums 8 logarithms of lengths of 1e-9 ... 2e-7 m (of size 20,
    # rounded to 1.8e-15 each) or 8 angles, over 4 pi, in either form; the
    # scaled coordinates round once more (1e-16 of offsets up to 100 edges)
    far = np.abs(g.centre[:, None] - g.centre[None])[..., 0] > 25e-9
    assert np.abs(got - ref)[far].max() < 5e-14
    assert np.linalg.norm((got - ref)[~far]) < 1e-12 * np.linalg.norm(ref[~far])
    if layers == 1:  # mirror symmetry
        assert np.abs(got[..., [2, 4]]).max() <= 1e-12


@pytest.mark.parametrize("cells,jitter", [((1, 1, 1), 0.0), ((4, 3, 2), 0.0), ((19, 1, 1), 0.2)])
def test_tetra_blocks(mt, ctx, cells, jitter):
    # 6 tiles; 144 (more than one 128-row group, 16-column groups whole); 114
    # (ragged groups, distances of up to 19 cells)
    verts, tets = wl.tetra_box(*cells, size=tuple(5e-9 * c for c in cells), jitter=jitter, seed=3)
    n = len(tets)
    tiles = mt.mt_tiles_create_tetra(ctx, verts, tets, 8e5, 1.3e-11, 0.0)
    ref = oracle.tetra_demag_tensor(verts[tets]).reshape(n, n, 6)
    got = mt.mt_tensor_read_rows(mt.mt_demag_assemble(tiles, "f64"), 0, n)
    assert np.linalg.norm(got - ref) < 1e-12 * np.linalg.norm(ref)
    # distant blocks are differences of angles and edge integrals of order
    # 0.1 ... 1 (round-off 1e-16 each, 26 of them)
    assert np.abs(got - ref).max() < 5e-15 + 1e-12 * np.abs(ref).max() * (jitter > 0)
    pairs = np.stack(np.meshgrid(np.arange(n), np.arange(n), indexing="ij"), -1).reshape(-1, 2)
    assert np.abs(mt.mt_demag_blocks(tiles, pairs).reshape(n, n, 6) - got).max() < 1e-15
