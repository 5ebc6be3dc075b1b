"""The fast Euler screens (wt_central.cuh) at the ends of FP32's range: gas so cold or thin that the products
with 1 / c^2 raise what the FP32 pairs lose below 2^-125 above the threshold under which theta does not
matter, and data whose indicators' squares pass 2^128."""
import numpy as np
import pytest

from paper_1504_00731_gb300 import workloads as W

torch = pytest.importorskip("torch")


def _check(b, O, flux, U, lens):
    P = O.problem(flux, bc=0, alpha_R=50.0)
    ref = O.rhs(P, U, *lens)
    grid = b.grid_1d(U.shape[1], 0.0, 1.0) if U.ndim == 2 else b.grid_2d(U.shape[2], U.shape[1])
    prob = b.problem(flux, alpha_R=50.0)
    ws = b.alloc_workspace(b.workspace_bytes(prob, grid))
    u = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    L = torch.empty_like(u)
    b.weno_theta_rhs(prob, grid, u, L, ws)
    ax = tuple(range(1, U.ndim))
    spread = np.max([np.abs(O.rhs(P, W.ulp_perturbed(U, s), *lens) - ref).max(axis=ax) for s in range(3)], axis=0)
    err = np.abs(L.cpu().numpy() - ref).max(axis=ax)
    assert np.all(err <= np.maximum(1e-13 * np.abs(ref).max(axis=ax), 10 * spread)), (err, spread)


@pytest.mark.gpu
@pytest.mark.parametrize("amp", [1e-9, 1e-10])
@pytest.mark.parametrize("a,c", [(-55, -28), (-40, -28), (-55, -20), (0, -28), (0, 0)])
@pytest.mark.parametrize("shape", [(700,), (20011,), (40, 50)])
def test_rhs_of_cold_and_thin_gas(wtlib, oracle, shape, a, c, amp):
    """Pressure noise in a uniform stream, density 2^a and sound speed about 2^c: RHS within 1e-13 of the largest
    |L| per component, or ten times the oracle's own spread over data moved by at most one ulp."""
    rng = np.random.default_rng(11)
    r, one = np.full(shape, 2.0**a), np.full(shape, 2.0**c)
    p = 2.0 ** (a + 2 * c) * (1 + amp * rng.uniform(-1, 1, shape))
    if len(shape) == 1:
        _check(wtlib, oracle, wtlib.WT_FLUX_EULER1D, W.cons_1d(r, one, p), (1.0 / shape[0],))
    else:
        _check(wtlib, oracle, wtlib.WT_FLUX_EULER2D, W.cons_2d(r, one, 0.5 * one, p), (1.0 / shape[1], 1.0 / shape[0]))


@pytest.mark.gpu
@pytest.mark.parametrize("k", [-2, -1, 0, 1, 2])
def test_rhs_2d_of_dense_fast_streams(wtlib, oracle, k):
    """Noise of 2^k in the transverse velocity of a stream with rho u = 2^60 beside one twice as fast (so that
    neither side of the splitting vanishes): the squares of the fourth differences' sums lie on
    both sides of 2^128.  The same bounds."""
    rng = np.random.default_rng(12)
    ny, nx = shape = (24, 600)
    u = np.where(np.arange(nx) < nx - 8, 2.0**10, 2.0**11) * np.ones(shape)
    U = W.cons_2d(np.full(shape, 2.0**50), u, 2.0**k * rng.uniform(-1, 1, shape), np.full(shape, 2.0**70))
    _check(wtlib, oracle, wtlib.WT_FLUX_EULER2D, U, (1.0 / nx, 1.0 / ny))
    V = np.ascontiguousarray(U[[0, 2, 1, 3]].transpose(0, 2, 1))
    _check(wtlib, oracle, wtlib.WT_FLUX_EULER2D, V, (1.0 / ny, 1.0 / nx))
