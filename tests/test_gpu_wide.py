"""Walk of the 32-wide boxes against the one-thread-per-particle walk (Alg. 1):
the same rows, entry for entry (both list a particle's neighbours tree by tree,
image by image, in Z-order), at the sizes where its nodes, its groups of 32
survivors and its lanes per particle change."""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_08088_gb300 import _lib
from paper_1901_08088_gb300.qbvh import NeighborList

pytestmark = pytest.mark.gpu


def _pos4(xyz, types=None):
    out = np.zeros((len(xyz), 4), np.float32)
    out[:, :3] = xyz
    if types is not None:
        out[:, 3] = np.asarray(types, np.int32).view(np.float32)
    return torch.from_numpy(out).cuda()


def _rows(pos4, off, Ls, r, T, cap, traversal, type_trees=1):
    nl = NeighborList()
    nl.set_option(_lib.QBVH_OPT_TRAVERSAL, traversal)
    nl.set_option(_lib.QBVH_OPT_TYPE_TREES, type_trees)
    if len(Ls) == 1:
        nl.build(pos4, Ls[0], T)
    else:
        nl.build_batched(pos4, off, Ls, T)
    rc = nl.query(r, cap=cap, max_retries=0, raise_on_error=False)
    rows, counts = nl.neighbors()
    rows, counts = rows.clone(), counts.clone()
    nl.close()
    live = torch.arange(rows.shape[1], device="cuda")[None, :] < counts[:, None]
    return rc, torch.where(live, rows, -1), counts


def _same(pos4, off, Ls, r, T=1, cap=256, type_trees=1):
    got = _rows(pos4, off, Ls, r, T, cap, 1, type_trees)
    ref = _rows(pos4, off, Ls, r, T, cap, 0, type_trees)
    assert got[0] == ref[0]
    assert torch.equal(got[2], ref[2])
    assert torch.equal(got[1], ref[1])


def _fluid(n, rho, seed):
    rng = np.random.default_rng(seed)
    L = np.float32((n / rho) ** (1 / 3))
    x = rng.uniform(0, float(L), (n, 3)).astype(np.float32)
    x[x >= L] = 0
    return x, float(L)


@pytest.mark.parametrize("n", [64, 65, 1023, 1024, 1025, 7999, 8000, 8007, 32767, 32769, 59999, 60000, 60031, 70001, 199999, 200001])
def test_sizes(n):
    x, L = _fluid(n, 0.6, n)
    _same(_pos4(x), [0, n], [L], min(2.2, 0.45 * L))


@pytest.mark.parametrize("n", [900, 9000, 65000])
@pytest.mark.parametrize("type_trees", [0, 1])
def test_types(n, type_trees):
    x, L = _fluid(n, 0.7, n)
    t = np.random.default_rng(1).integers(0, 3, n)
    r = np.full((3, 3), 1.9, np.float32)
    if type_trees:
        r = np.array([[1.9, 1.4, 0.0], [1.4, 2.3, 1.0], [0.0, 1.0, 1.2]], np.float32)
    _same(_pos4(x, t), [0, n], [L], r, T=3, type_trees=type_trees)


def test_batched_uneven():
    ns = [1, 40, 0, 33, 1500, 31, 20000, 7, 45000, 2]
    xs, Ls = zip(*[_fluid(max(n, 300), 0.6, 7 + k) for k, n in enumerate(ns)])
    xs = [x[:n] for x, n in zip(xs, ns)]
    _same(_pos4(np.concatenate(xs)), np.concatenate([[0], np.cumsum(ns)]), Ls, 2.0)


@pytest.mark.parametrize("m", [16, 24, 40])
def test_pairs_at_the_radius(m):
    """A lattice of spacing 1/2 whose shells lie exactly at the radius, inside the
    box and across its faces: every group of survivors holds such a pair."""
    g = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.float32) * 0.5
    for r in (1.5, np.nextafter(np.float32(1.5), np.float32(2)), np.nextafter(np.float32(1.5), np.float32(1))):
        _same(_pos4(g), [0, len(g)], [0.5 * m], float(r))
    # and rounded coordinates, whose shells scatter around the radius
    L = np.float32(0.3 * m)
    h = (g * 2 * np.float32(0.3)).astype(np.float32)
    h[h >= L] = 0
    _same(_pos4(h), [0, len(h)], [float(L)], 0.9)


@pytest.mark.parametrize("n", [5000, 20000, 65000])
def test_rows_past_the_capacity(n):
    x, L = _fluid(n, 0.7, 3)
    _same(_pos4(x), [0, n], [L], 2.4, cap=24)


@pytest.mark.parametrize("n", [3000, 64000])
def test_one_cluster(n):
    """Every particle near one point at a box corner: all images, long rows."""
    rng = np.random.default_rng(5)
    x = np.mod(rng.normal(0, 1.2 if n < 10000 else 6.0, (n, 3)), 60.0).astype(np.float32)
    x[x >= 60.0] = 0
    _same(_pos4(x), [0, n], [60.0], 0.6, cap=2048)


@pytest.mark.parametrize("n", [4099, 20003, 65003])
def test_double_precision_last_packet(n):
    """Double-precision data whose last packet has idle lanes, pairs at the radius
    near the box corner where those lanes' zero positions lie."""
    rng = np.random.default_rng(n)
    L = float((n / 0.6) ** (1 / 3))
    x = rng.uniform(0, L, (n, 3))
    r = np.float32(1.75)
    k = min(64, n)
    d = rng.normal(size=(k, 3))
    x[:k] = np.mod(float(r) * (1 + 1e-9 * rng.integers(-2, 3, (k, 1))) * d / np.linalg.norm(d, axis=1, keepdims=True), L)
    x[k] = 0.0
    x[x >= L] = 0.0
    pos = torch.from_numpy(np.concatenate([x, np.zeros((n, 1))], 1)).cuda()
    nl = NeighborList()
    nl.build_f64(pos, L, 1).query(float(r), cap=128)
    rows, counts = (v.cpu().numpy() for v in nl.neighbors())
    nl.close()
    ro, co = oracle.nlist64(x, L, r, cap=rows.shape[1])
    assert np.array_equal(counts, co)
    big = np.iinfo(np.int32).max
    live = np.arange(rows.shape[1])[None, :] < counts[:, None]
    assert np.array_equal(np.sort(np.where(live, rows, big), 1), np.sort(np.where(live, ro[:, :rows.shape[1]], big), 1))
