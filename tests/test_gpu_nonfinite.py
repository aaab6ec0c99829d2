"""States that are not finite are reported in the status word by every call that computes fluxes, also
where the whole stencil is alike (the FP32 screen must not take it for a constant one)."""
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


@pytest.mark.parametrize("K", [6, 8])
@pytest.mark.parametrize("shape,bc", [((300,), (1,)), ((5000,), (0,)), ((40, 30), (0, 1)), ((14, 15, 16), (0, 0, 1))])
def test_states_without_a_finite_value_are_reported(T, shape, bc, K):
    S = T.Solver(shape, tuple(1.0 / n for n in shape), bc, T.make_scheme(K))
    prim = PB.random_state(tuple(reversed(shape)), 3, jumps=False)
    U0 = S.init_state(torch.from_numpy(np.ascontiguousarray(prim)).cuda())
    dt = torch.full((1,), 1e-4, dtype=torch.float64, device="cuda")
    for kind in ("nan", "energy inf"):
        U = U0.clone()
        if kind == "nan":
            U.fill_(float("nan"))
        else:
            U[-1].fill_(float("inf"))
        out = torch.empty_like(U)
        S.rhs(U, out=out)
        assert S.status(reset=True) & T.ST_NONFINITE, kind
        S.face_dump(U, 0)
        assert S.status(reset=True) & T.ST_NONFINITE, kind
        S.rk3_step(U.clone(), dt)
        assert S.status(reset=True) & T.ST_NONFINITE, kind
        S.rhs_record(U, S.new_lin(), out=out)
        assert S.status(reset=True) & T.ST_NONFINITE, kind
        S.advance(U.clone(), 1)
        st = S.status(reset=True)
        assert st & T.ST_NONFINITE, kind
        if kind == "nan":
            assert st & T.ST_RHO and st & T.ST_P
    S.close()


@pytest.mark.parametrize("K", [6, 8])
def test_sound_speeds_whose_square_leaves_the_fast_division(T, K):
    """c^2 above 2^126, where the fast division returns 0: a pressure step in a smooth flow must still be
    seen.  Tolerance as for every filtered-against-FP64 comparison of fluxes: 1e-13 of the largest."""
    nx, ny = 64, 8
    i = np.arange(nx) + 0.5
    c = 1.2e19
    prim = np.empty((4, ny, nx))
    prim[0] = 1.0
    prim[1] = 0.1 * c + 2e-4 * c * np.sin(2.0 * np.pi * i / nx)
    prim[2] = 0.0
    prim[3] = c * c / 1.4 * np.where((i > 20) & (i < 44), 1.0 + 5e-5, 1.0)
    F = []
    for dec in (T.DECIDE_FILTERED, T.DECIDE_FP64):
        S = T.Solver((nx, ny), (1.0, 1.0), (0, 0), T.make_scheme(K, decisions=dec))
        U = S.init_state(torch.from_numpy(prim).cuda())
        F.append(S.face_dump(U, 0, flags=False)[0].cpu().numpy())
        S.close()
    for v in range(4):
        big = max(np.abs(F[1][v]).max(), 1e-2 * c * np.abs(F[1][0]).max() if v else 0.0)
        assert np.abs(F[0][v] - F[1][v]).max() <= 1e-13 * big, v
