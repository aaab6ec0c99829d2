"""Short 1D grids advance in one launch of one cluster: its steps against the same SSP-RK3 step
built from the operator calls (the grid sweeps), at the shortest lines, around the cluster's
shares and at both sides of the size where the grid path takes over."""
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


@pytest.mark.parametrize("n", [4, 17, 63, 64, 65, 255, 1919, 1920, 1921, 1952, 1953])
@pytest.mark.parametrize("K,lim,bc", [(6, 0, 1), (8, 1, 0), (8, 0, 1), (6, 2, 0)])
def test_line_steps_equal_operator_steps(T, n, K, lim, bc):
    """Three steps, each component to 1e-13 of its largest value: the two paths round the same
    sums in another order, and a decision that rounding sets moves a value at rounding level."""
    prim = PB.random_state((n,), 5 * n + K + lim, jumps=n > 32)
    S = T.Solver((n,), (1.0 / n,), (bc,), T.make_scheme(K, limiter=lim))
    U = S.init_state(torch.from_numpy(prim).cuda())
    V = U.clone()
    t = torch.zeros(1, dtype=torch.float64, device="cuda")
    S.advance(U, 3, t_dev=t)
    total = 0.0
    for _ in range(3):
        dt = S.max_dt(V, 0.4).item()
        V1 = V + dt * S.rhs(V)
        V2 = 0.75 * V + 0.25 * (V1 + dt * S.rhs(V1))
        V = V / 3.0 + 2.0 / 3.0 * (V2 + dt * S.rhs(V2))
        total += dt
    got, want = U.cpu().numpy(), V.cpu().numpy()
    for v in range(3):
        np.testing.assert_allclose(got[v], want[v], rtol=0, atol=1e-13 * np.abs(want).max())
    assert abs(t.item() - total) <= 1e-13 * total
    assert S.status() == 0
    S.close()


def test_line_stops_at_t_end_and_steps_with_given_dt(T):
    """The last step is clipped to t_end, later ones change nothing bit for bit; rk3_step with the
    same dt gives the same step."""
    n = 300
    prim, dx = PB.riemann_1d(n, 9)
    S = T.Solver((n,), (dx,), (1,), T.make_scheme(6))
    U = S.init_state(torch.from_numpy(prim).cuda())
    W = U.clone()
    dt = S.max_dt(U, 0.4).clone()
    t = torch.zeros(1, dtype=torch.float64, device="cuda")
    t_end = 2.5 * dt.item()
    S.advance(U, 600, t_end=t_end, t_dev=t)  # more than one launch's steps
    assert t.item() == t_end
    V = U.clone()
    S.advance(V, 3, t_end=t_end, t_dev=t)
    assert torch.equal(U, V) and t.item() == t_end
    X = W.clone()
    S.rk3_step(W, dt)
    S.t.zero_()
    S.advance(X, 1)
    assert torch.equal(W, X)
    S.close()
