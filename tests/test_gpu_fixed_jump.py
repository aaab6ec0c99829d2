"""Face fluxes beside strong jumps: a face whose stencil reaches across a jump must not carry the
rounding of the values beyond it (the nonlinear kernel adds limiter corrections to the central
flux, which does hold them; such items take the FP64 reconstruction instead)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

REACH = [(-1, 1), (0, 2), (-2, 0), (0, 3), (-3, 0), (0, 4)]  # cells i + j of candidate k (Table 1)


def reaches_jump(flags, rho, K, ax):
    """Faces with a smooth candidate (delta_k = 1) on a cell of more than twice the density of the
    face's own two: its far values belong to the face value."""
    n = rho.shape[ax]
    own = np.maximum(np.roll(rho, 1, axis=ax), rho)
    over = np.zeros(rho.shape, dtype=bool)
    for side in range(2):
        for k in range(K - 2):
            kept = np.take((flags[..., side] >> k & 1).any(axis=-1), np.arange(n), axis=ax)
            for j in range(REACH[k][0], REACH[k][1] + 1):
                # face f: f_i is cell f - 1; f- has it mirrored, f_i is cell f
                far = np.roll(rho, 1 - j if side == 0 else j, axis=ax) > 2.0 * own
                over |= kept & far
    return np.concatenate([over, np.take(over, [0], axis=ax)], axis=ax)


@pytest.mark.parametrize("K", [6, 8])
@pytest.mark.parametrize("ratio", [30.0, 1000.0])
@pytest.mark.parametrize("spikes", [False, True])
def test_flux_beside_jumps_has_the_rounding_of_its_own_cells(orc, K, ratio, spikes):
    """Density and pressure jump by `ratio` every 7 cells (or in one cell of 9) of a rough field; TVD5,
    which puts a value of the nearest cells in the place of a candidate (the MP median x + minmod(a - x,
    b - x) rounds at the size of the candidate x that it replaces, in every evaluation).
    Tolerance: both evaluations round sums of at most about 100 terms of the size of the face's
    two cells' |lambda U| where no smooth candidate reaches beyond the jump: 100 u (300-600 u when the
    far values' rounding stays)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2010_13289_gb300 import tenom as T
    lim = 1
    rng = np.random.default_rng(int(K + ratio))
    nx, ny = 210, 36
    for axis in (0, 1):
        prim = np.stack([1.0 + 0.05 * rng.standard_normal((ny, nx)), 0.1 * rng.standard_normal((ny, nx)),
                         0.1 * rng.standard_normal((ny, nx)), 1.0 + 0.05 * rng.standard_normal((ny, nx))])
        i = np.arange(nx) if axis == 0 else np.arange(ny)[:, None]
        m = (i % 9 == 4) if spikes else (i // 7 % 2 == 1)
        prim[0] = np.where(m, prim[0] * ratio, prim[0])
        prim[3] = np.where(m, prim[3] * ratio, prim[3])
        shape, dx, bc = (nx, ny), (1.0 / nx, 1.0 / ny), (0, 0)
        S = T.Solver(shape, dx, bc, T.make_scheme(K, limiter=lim))
        g, so = orc.make_grid(shape, dx, bc), orc.make_scheme(K, limiter=lim)
        U = orc.init_state(g, prim)
        Fg, flg = S.face_dump(torch.from_numpy(U).cuda(), axis)
        Fo, flo = orc.faces(g, so, U, axis)[:2]
        same = (flg.cpu().numpy() == flo).all(axis=(-2, -1))
        assert same.mean() > 0.99
        same &= ~reaches_jump(flo, prim[0], K, 1 - axis)
        assert same.mean() > 0.3
        rho, E = U[0], U[3]
        p = 0.4 * (E - 0.5 * (U[1] ** 2 + U[2] ** 2) / rho)
        c = np.sqrt(1.4 * p / rho)
        lam = np.abs(U[1 + axis] / rho) + c
        cell = np.stack([lam * rho, lam * rho * (c + lam), lam * rho * (c + lam), lam * (E + p)])
        ax = 2 - axis
        near = np.maximum(np.roll(cell, 1, axis=ax), cell)  # face f lies between cells f - 1 and f
        near = np.concatenate([near, np.take(near, [0], axis=ax)], axis=ax)
        err = (np.abs(Fg.cpu().numpy() - Fo) / near)[:, same] * 2.0 ** 53
        assert err.max() <= 100.0, (axis, err.max(axis=1))
        assert S.status() == 0
        S.close()
