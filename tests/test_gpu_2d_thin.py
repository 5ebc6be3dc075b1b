"""2D grids with more rows of tiles than the y dimension of a launch holds (65535: the fast tiles have 7 rows,
the strict ones 8)."""
import numpy as np
import pytest

from paper_1504_00731_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("strict,ny", [(False, 458745), (False, 458746), (True, 524281)])
def test_thin_grid(wtlib, oracle, strict, ny):
    """3 x ny cells: RHS against the oracle (bit for bit in strict mode; else within 1e-13 of the largest |L|
    or ten times the oracle's own spread), and two steps equal to one and one."""
    b, O = wtlib, oracle
    nx = 3
    y = (np.arange(ny) + 0.5) / ny
    col = lambda v: np.repeat(v[:, None], nx, axis=1)  # noqa: E731
    U = W.cons_2d(col(1 + 0.2 * np.sin(40 * y)), col(0.1 * np.cos(30 * y)), col(0.3 + 0.1 * np.sin(50 * y)),
                  col(np.where((y > 0.4) & (y < 0.999), 1.0, 0.4)))
    U[0, :, 1] += 0.01
    dx, dy = 1.0 / nx, 1.0 / ny
    P = O.problem(O.FLUX_EULER2D, bc=0, alpha_R=10.0)
    ref = O.rhs(P, U, dx, dy)
    g = b.grid_2d(nx, ny)
    prob = b.problem(b.WT_FLUX_EULER2D, alpha_R=10.0, mode=b.WT_MODE_STRICT if strict else b.WT_MODE_FAST)
    ws = b.alloc_workspace(b.workspace_bytes(prob, g))
    u = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    L = torch.empty_like(u)
    b.weno_theta_rhs(prob, g, u, L, ws)
    got = L.cpu().numpy()
    if strict:
        assert np.array_equal(got, ref)
    else:
        spread = np.max([np.abs(O.rhs(P, W.ulp_perturbed(U, s), dx, dy) - ref).max(axis=(1, 2)) for s in range(3)], axis=0)
        assert np.all(np.abs(got - ref).max(axis=(1, 2)) <= np.maximum(1e-13 * np.abs(ref).max(axis=(1, 2)), 10 * spread))
    v, w = u.clone(), u.clone()
    t2, _ = b.weno_theta_step(prob, g, v, 0.4, ws, max_steps=2)
    ta, _ = b.weno_theta_step(prob, g, w, 0.4, ws, max_steps=1)
    tb, _ = b.weno_theta_step(prob, g, w, 0.4, ws, max_steps=1)
    assert torch.equal(v, w) and t2 == ta + tb
