"""The fast policy's screened scalar tiles (scalar_fluxes in wt_kernels.cuh) against the oracle, and every
launch path against the others bit for bit.

The screen decides theta (Eq. (tau_we6)) in FP32, which holds nothing below 2^-149: data whose
differences, or their products with alpha, lie there must be left to FP64.  For advection off the
unit speed one side of the splitting is zero and is dropped."""
import numpy as np
import pytest

from paper_1504_00731_gb300 import workloads as W

torch = pytest.importorskip("torch")


def _state(kind, n):
    x = (np.arange(n) + 0.5) / n
    wave = 0.3 + np.sin(2 * np.pi * x)
    if kind == "smooth":
        u = wave
    elif kind == "shock":
        u = np.where(x < 0.4, 1.25, -0.5) + 0.1 * wave
    elif kind == "noise":
        return W.ulp_perturbed(np.full((1, n), 0.7), 3)
    elif kind == "rough":
        u = np.random.default_rng(5).uniform(-1.0, 1.0, n)
    elif kind == "large":  # beyond the screen's range
        u = wave * 2.0**62
    elif kind == "tails":  # a pulse whose tails run through every binade down to zero
        u = np.exp(-(40.0 * (x - 0.5)) ** 2)
    else:  # "step 2^k": two levels, and a wave, of that size
        A = 2.0 ** int(kind.split("^")[1])
        u = np.where(x < 0.3, A, 0.0) + np.where((x > 0.5) & (x < 0.9), A * (1 + 0.2 * np.sin(40 * x)), 0.0)
    return u[None, :]


KINDS = ["smooth", "shock", "noise", "rough", "large", "tails", "step 2^-20", "step 2^-50", "step 2^-80", "step 2^-130"]


def _check(b, O, flux, a, kind, n):
    u = _state(kind, n)
    P = O.problem(flux, adv_speed=a, bc=O.BC_OUTFLOW, alpha_R=10.0)
    ref = O.rhs(P, u, 1.0 / n)
    g = b.grid_1d(n, 0.0, 1.0)
    prob = b.problem(flux, adv_speed=a, bc=b.WT_BC_OUTFLOW, alpha_R=10.0)
    ws = b.alloc_workspace(b.workspace_bytes(prob, g))
    u0 = torch.from_numpy(np.ascontiguousarray(u)).cuda()
    L = torch.empty_like(u0)
    b.weno_theta_rhs(prob, g, u0, L, ws)
    spread = max(np.abs(O.rhs(P, W.ulp_perturbed(u, s), 1.0 / n) - ref).max() for s in range(3))
    assert np.abs(L.cpu().numpy() - ref).max() <= max(1e-13 * np.abs(ref).max(), 10 * spread)
    return prob, g, ws, u0


@pytest.mark.gpu
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("flux,a", [("advection", 1.0), ("advection", 0.3), ("advection", -1.7), ("burgers", 1.0)])
@pytest.mark.parametrize("n", [3, 62, 64, 127, 128, 700, 7753, 20011])
def test_screened_scalar_fluxes(wtlib, oracle, kind, flux, a, n, monkeypatch):
    """RHS within 1e-13 of the largest |L|, or ten times the oracle's own spread over data moved by at most
    one ulp; three steps the same bits through the persistent kernels, the stage kernels and both
    batched tiles."""
    b = wtlib
    code = b.WT_FLUX_ADVECTION if flux == "advection" else b.WT_FLUX_BURGERS
    prob, g, ws, u0 = _check(b, oracle, code, a, kind, n)
    runs = []
    for launch in (b.WT_LAUNCH_AUTO, b.WT_LAUNCH_STAGES):
        pl = b.problem(code, adv_speed=a, bc=b.WT_BC_OUTFLOW, alpha_R=10.0, launch=launch)
        u = u0.clone()
        b.weno_theta_step(pl, g, u, 0.4, ws, max_steps=3)
        runs.append(u)
    s = b.WtSegment()
    s.offset, s.n, s.lo, s.hi, s.bc_lo, s.bc_hi = 0, n, 0.0, 1.0, b.WT_BC_OUTFLOW, b.WT_BC_OUTFLOW
    wb = b.alloc_workspace(b.workspace_bytes(prob, None, n, 1))
    for tile in (63, 127):
        monkeypatch.setenv("WT_BATCHED_TILE", str(tile))
        u = u0.clone()
        b.weno_theta_step_batched(prob, [s], u, n, 0.4, 3, wb)
        runs.append(u)
    for r in runs[1:]:
        assert torch.equal(r, runs[0])
