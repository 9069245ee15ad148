"""The LJ pass at the sizes where its blocks' rounds, its lanes per particle and
its row chunks end, against the FP64 oracle on the same list."""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_08088_gb300 import _lib
from paper_1901_08088_gb300.qbvh import NeighborList, check, qbvh_lj_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [65, 127, 129, 3001, 29999, 30001])
@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("lanes", [None, 1, 8])
@pytest.mark.parametrize("grad", [False, True])
def test_rounds(n, T, lanes, grad):
    rng = np.random.default_rng(n + T)
    m = int(np.ceil(n ** (1 / 3)))
    L = np.float32(m * 1.1)
    ijk = np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    x = np.mod((ijk + 0.5) * 1.1 + 0.15 * rng.uniform(-1, 1, (n, 3)), float(L)).astype(np.float32)
    x[x >= L] = 0
    t = rng.integers(0, T, n).astype(np.int32)
    r_cut = np.float32(min(2.1, 0.45 * float(L)))
    pos4 = np.concatenate([x, t.view(np.float32)[:, None]], 1)
    pos4 = torch.from_numpy(np.ascontiguousarray(pos4)).cuda()
    eps = np.array([[1.0, 1.5], [1.5, 0.5]], np.float32)[:T, :T].copy()
    sig = np.array([[1.0, 0.88], [0.88, 0.8]], np.float32)[:T, :T].copy()
    nl = NeighborList()
    if lanes is not None:
        nl.set_option(_lib.QBVH_OPT_LJ_LANES, lanes)
    nl.build(pos4, float(L), T).query(float(r_cut), cap=64)
    rows, counts = (v.cpu().numpy() for v in nl.neighbors())
    e, F = torch.empty(n, device="cuda"), torch.empty((n, 3), device="cuda")
    U = torch.empty(1, device="cuda", dtype=torch.float64)
    dE = torch.empty((T, T), device="cuda", dtype=torch.float64) if grad else None
    dS = torch.empty((T, T), device="cuda", dtype=torch.float64) if grad else None
    check(qbvh_lj_forward(nl.h, pos4, torch.from_numpy(eps).cuda(), torch.from_numpy(sig).cuda(),
                          np.full((T, T), r_cut, np.float32), e, U, F, dE, dS), "qbvh_lj_forward")
    torch.cuda.synchronize()
    ref = oracle.lj_fp64(x, t, float(L), eps, sig, np.full((T, T), r_cut, np.float32), rows, counts)
    # FP32 sums of at most 64 terms: 1e-5 relative (the library's stated bound)
    assert abs(U.item() - ref["U"]) <= 1e-5 * abs(ref["U"])
    assert np.linalg.norm(F.cpu().numpy() - ref["F"]) <= 1e-5 * np.linalg.norm(ref["F"])
    assert abs(float(e.double().sum()) - ref["U"]) <= 1e-5 * abs(ref["U"])
    if grad:
        assert np.allclose(dE.cpu().numpy(), ref["dE"], rtol=1e-5, atol=0)
        assert np.allclose(dS.cpu().numpy(), ref["dS"], rtol=1e-5, atol=0)
    nl.close()


def _pass(nl, pos4, T, r_cut):
    """U, dU/deps, dU/dsig of the handle's systems with every eps and sigma one."""
    S = nl.n_sys
    one = torch.ones((T, T), device="cuda")
    U = torch.empty(S, device="cuda", dtype=torch.float64)
    dE, dS = (torch.empty((S, T, T), device="cuda", dtype=torch.float64) for _ in range(2))
    check(qbvh_lj_forward(nl.h, pos4, one, one, np.full((T, T), r_cut, np.float32), None, U, None, dE, dS),
          "qbvh_lj_forward")
    return U.cpu().numpy(), dE.cpu().numpy(), dS.cpu().numpy()


@pytest.mark.parametrize("lanes", [None, 1, 2, 4, 8, 16, 32])
def test_gradient_terms_enter_fp64_per_lane(lanes):
    """With eps = 1 a lane's FP32 sum of dU/deps terms is its FP32 sum of energies,
    so both FP64 totals add the same numbers: equal up to FP64 roundings (32,768
    particles of up to 32 lanes, sums of one sign: 1e-12).  One FP32 rounding per
    particle on the way would show as about 2^-24 / sqrt(32,768) = 3e-10."""
    n, r_cut = 32768, np.float32(2.5)
    rng = np.random.default_rng(4)
    ijk = np.stack(np.meshgrid(*[np.arange(32)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = ((ijk + 0.5) * 1.1 + 0.08 * rng.uniform(-1, 1, (n, 3))).astype(np.float32)
    pos4 = torch.from_numpy(np.concatenate([x, np.zeros((n, 1), np.float32)], 1)).cuda()
    nl = NeighborList()
    if lanes is not None:
        nl.set_option(_lib.QBVH_OPT_LJ_LANES, lanes)
    nl.build(pos4, 35.2, 1).query(float(r_cut), cap=96)
    U, dE, _ = _pass(nl, pos4, 1, r_cut)
    nl.close()
    assert abs(dE[0, 0, 0] - U[0]) <= 1e-12 * abs(U[0])


@pytest.mark.parametrize("T", [1, 2, 3])
def test_gradient_terms_of_a_cluster(T):
    """Nine particles in reach of one another: with eight lanes per particle every
    lane holds one pair, so the totals are those of the 36 pairs, each computed as a
    system of its own, added in FP64 (36 terms: 1e-14 of their sizes)."""
    rng = np.random.default_rng(8)
    g = np.stack(np.meshgrid(*[np.arange(3)] * 2, indexing="ij"), -1).reshape(-1, 2)
    x = np.concatenate([g, np.zeros((9, 1))], 1) * 1.05 + 0.08 * rng.uniform(-1, 1, (9, 3)) + 9.0
    t = rng.integers(0, T, 9).astype(np.int32)
    p = np.concatenate([x.astype(np.float32), t.view(np.float32)[:, None]], 1)
    i, j = np.triu_indices(9, 1)
    pairs = np.stack([p[i], p[j]], 1).reshape(-1, 4)
    got = []
    for q, S in ((p, 1), (pairs, 36)):
        q = torch.from_numpy(np.ascontiguousarray(q)).cuda()
        nl = NeighborList()
        nl.build_batched(q, np.arange(S + 1) * (len(q) // S), [20.0] * S, T).query(4.0, cap=8)
        assert int(nl.neighbors()[1].min()) == (8 if S == 1 else 1)
        got.append(_pass(nl, q, T, np.float32(4.0))[1:])
        nl.close()
    for whole, parts in zip(*got):
        assert np.all(np.abs(whole[0] - parts.sum(0)) <= 1e-14 * np.abs(parts).sum(0))
