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
