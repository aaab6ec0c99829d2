"""The 1D tile code against steps that do not use it: short-line launches and the batched launch against
SSP-RK3 steps built from the operator, the CFL call and the positivity limiter, and 1D screen tiles at
their edges against FP64 decisions."""
import numpy as np
import pytest

from paper_2010_13289_gb300 import problems as PB

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2010_13289_gb300 import tenom
    tenom.lib()
    return tenom


def operator_step(S, U, dt, dx, pp):
    """One step from face fluxes (limited when pp), as the grid sweeps compute them."""
    dt_dev = torch.full((1,), dt, dtype=torch.float64, device="cuda")

    def euler(V):
        F = S.face_dump(V, 0, flags=False)[0]
        if pp:
            S.positivity_limit(V, 0, dt_dev, F)
        return V - dt / dx * (F[:, 1:] - F[:, :-1])
    V = euler(U)
    V = 0.75 * U + 0.25 * euler(V)
    return U / 3.0 + 2.0 / 3.0 * euler(V)


def close(got, want):
    """1e-13 of each component's largest: the same sums in another order (tests of the line launch)."""
    for v in range(3):
        big = max(want[v].abs().max().item(), 1e-3 * want.abs().max().item())
        assert (got[v] - want[v]).abs().max().item() <= 1e-13 * big, v


@pytest.mark.parametrize("n", [1, 2, 3, 33, 45, 60, 300])
@pytest.mark.parametrize("K,lim,pp", [(6, 0, 0), (8, 1, 0), (6, 1, 1), (8, 0, 1)])
def test_line_steps_with_and_without_the_limiter(T, n, K, lim, pp):
    """Sizes of every cluster width, the smallest lines (transmissive), and the limiter (it changes faces of
    no smooth state: its decisions are the same on both sides)."""
    prim = PB.random_state((max(n, 8),), 3 * n + K, jumps=n > 8)[:, :n].copy()
    dx = 1.0 / n
    S = T.Solver((n,), (dx,), (1,), T.make_scheme(K, limiter=lim, positivity=pp))
    U = S.init_state(torch.from_numpy(np.ascontiguousarray(prim)).cuda())
    V = U.clone()
    for _ in range(2):
        dt = S.max_dt(V, 0.3).item()
        V = operator_step(S, V, dt, dx, pp)
    S.advance(U, 2, cfl=0.3)
    close(U, V)
    assert S.status() == 0
    S.close()


@pytest.mark.parametrize("K,lim,pp,kw", [(6, 0, 0, {}), (8, 1, 0, {}), (8, 0, 1, {}), (6, 1, 1, {"decisions": 1}),
                                         (6, 0, 0, {"d": (0.4, 0.3, 0.1, 0.2)}), (8, 0, 0, {"decisions": 1})])
@pytest.mark.parametrize("tile", [64, 128, 256])
def test_batch_steps_equal_operator_steps(T, K, lim, pp, kw, tile):
    sizes = np.array([5, 63, 64, 127, 128, 255, 300], dtype=np.int32)
    scheme = T.make_scheme(K, limiter=lim, positivity=pp, **kw)
    prims = [PB.random_state((max(int(n), 8),), int(n) + K, jumps=n > 8)[:, :n] for n in sizes]
    dxs = 1.0 / sizes
    B = T.Batch(sizes, dxs, scheme)
    B.set_tiling(tile, 2)
    U = B.init_state(torch.from_numpy(np.ascontiguousarray(np.concatenate(prims, axis=1))).cuda())
    U0 = U.clone()
    B.step(U, 1, cfl=0.3)
    for j, n in enumerate(sizes):
        n = int(n)
        S = T.Solver((n,), (dxs[j],), (1,), scheme)
        V = U0[:, B.off[j]:B.off[j + 1]].contiguous()
        dt = S.max_dt(V, 0.3).item()
        close(U[:, B.off[j]:B.off[j + 1]], operator_step(S, V, dt, dxs[j], pp))
        S.close()
    assert B.status() == 0
    B.close()


@pytest.mark.parametrize("n,bc", [(127, 1), (128, 0), (128, 1), (129, 0), (256, 1), (257, 0)])
@pytest.mark.parametrize("K", [6, 8])
def test_1d_screen_tiles_at_their_edges(T, n, bc, K):
    """1D screen tiles hold 128 faces (tolerance as for the larger grids' comparison: 1e-13 of the largest)."""
    prim = PB.random_state((n,), n + K, jumps=True)
    F = []
    for dec in (T.DECIDE_FILTERED, T.DECIDE_FP64):
        S = T.Solver((n,), (1.0 / n,), (bc,), T.make_scheme(K, decisions=dec))
        F.append(S.face_dump(S.init_state(torch.from_numpy(prim).cuda()), 0, flags=False)[0])
        assert S.status() == 0
        S.close()
    close(F[0], F[1])
