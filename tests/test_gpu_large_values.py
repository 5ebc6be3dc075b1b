"""Fast-mode reconstructions of large data: the weights' common denominator prod_l (eps + beta_l) is formed of
scaled indicators where it would overflow."""
import numpy as np
import pytest

from paper_1504_00731_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [40, 700, 20011])
@pytest.mark.parametrize("k", [40, 44, 46, 50, 62, 70, 100])
@pytest.mark.parametrize("flux", ["advection", "burgers", "euler"])
def test_rhs_of_large_values(wtlib, oracle, flux, k, n):
    """Within 1e-13 of the largest |L| per component, or ten times the oracle's own spread over data moved by at
    most one ulp; a jump, so that the nonlinear weights are taken."""
    b, O = wtlib, oracle
    x = (np.arange(n) + 0.5) / n
    u = (np.where(x < 0.4, 1.25, -0.5) + 0.1 * np.sin(6 * x))[None, :]
    if flux == "euler":  # densities and energies (beta about 2^(2 k))
        u = W.cons_1d(np.where(x < 0.4, 1.0, 0.125), 0.1 * np.sin(6 * x), np.where(x < 0.4, 1.0, 0.1))
    u = u * 2.0**k
    code = {"advection": b.WT_FLUX_ADVECTION, "burgers": b.WT_FLUX_BURGERS, "euler": b.WT_FLUX_EULER1D}[flux]
    P = O.problem(code, bc=O.BC_OUTFLOW, alpha_R=10.0)
    ref = O.rhs(P, u, 1.0 / n)
    g = b.grid_1d(n, 0.0, 1.0)
    prob = b.problem(code, bc=b.WT_BC_OUTFLOW, alpha_R=10.0)
    ws = b.alloc_workspace(b.workspace_bytes(prob, g))
    u0 = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    L = torch.empty_like(u0)
    b.weno_theta_rhs(prob, g, u0, L, ws)
    spread = np.max([np.abs(O.rhs(P, W.ulp_perturbed(u, s), 1.0 / n) - ref).max(axis=1) for s in range(3)], axis=0)
    err = np.abs(L.cpu().numpy() - ref).max(axis=1)
    assert np.all(err <= np.maximum(1e-13 * np.abs(ref).max(axis=1), 10 * spread))
