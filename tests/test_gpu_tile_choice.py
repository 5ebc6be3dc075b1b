"""Fast 1D Euler grids of more than one tile per SM: step calls take 31-cell, then 63-cell resident tiles while these
are co-resident, then stage launches of 63-cell tiles, from 76,609 cells on of 127-cell tiles with six items
per thread; RHS calls change to the latter at 38,305 cells."""
import numpy as np
import pytest

from paper_1504_00731_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [4105, 4713, 9001, 14136, 14137, 28728, 28729, 38304, 38305, 45011, 76608, 76609, 80021])
def test_long_grids(wtlib, oracle, n, monkeypatch):
    """RHS against the oracle (1e-13 of the largest |L|, or ten times its spread over data moved by at most one
    ulp); three steps the same bits by the step call and by the batched tiles of 31, 63 and 127 cells."""
    b, O = wtlib, oracle
    x, _ = W.grid_1d(n, -5.0, 5.0, periodic=False)
    U = W.cons_1d(np.where(x < 0.3, 3.8, 1 + 0.2 * np.sin(5 * x)), np.where(x < 0.3, 2.6, 0.0), np.where(x < 0.3, 10.3, 1.0))
    U[:, ::4001] *= 1.5  # isolated jumps, so that tiles all over the grid hold listed interfaces
    dx = 10.0 / n
    P = O.problem(O.FLUX_EULER1D, bc=O.BC_OUTFLOW, alpha_R=10.0)
    ref = O.rhs(P, U, dx)
    g = b.grid_1d(n, -5.0, 5.0)
    prob = b.problem(b.WT_FLUX_EULER1D, bc=b.WT_BC_OUTFLOW, alpha_R=10.0)
    ws = b.alloc_workspace(b.workspace_bytes(prob, g))
    u0 = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    L = torch.empty_like(u0)
    b.weno_theta_rhs(prob, g, u0, L, ws)
    spread = np.max([np.abs(O.rhs(P, W.ulp_perturbed(U, s), dx) - ref).max(axis=1) for s in range(3)], axis=0)
    assert np.all(np.abs(L.cpu().numpy() - ref).max(axis=1) <= np.maximum(1e-13 * np.abs(ref).max(axis=1), 10 * spread))
    u = u0.clone()
    b.weno_theta_step(prob, g, u, 0.5, ws, max_steps=3)
    s = b.WtSegment()
    s.offset, s.n, s.lo, s.hi, s.bc_lo, s.bc_hi = 0, n, -5.0, 5.0, b.WT_BC_OUTFLOW, b.WT_BC_OUTFLOW
    wb = b.alloc_workspace(b.workspace_bytes(prob, None, n, 1))
    for code in (31, 63, 127, 5127):
        monkeypatch.setenv("WT_BATCHED_TILE", str(code))
        v = u0.clone()
        b.weno_theta_step_batched(prob, [s], v, n, 0.5, 3, wb)
        assert torch.equal(v, u), code
