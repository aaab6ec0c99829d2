"""Face timing covers the steps of short 1D grids too, and does not change them."""
import pytest

from paper_2010_13289_gb300 import problems as PB

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [40, 256, 1900])
def test_kernel_timing_counts_the_sweeps_of_short_lines(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2010_13289_gb300 import tenom as T
    prim, dx = PB.riemann_1d(n, 4)
    S = T.Solver((n,), (dx,), (1,), T.make_scheme(8))
    U = S.init_state(torch.from_numpy(prim).cuda())
    plain = S.advance(U.clone(), 2)
    S.kernel_timing(True)
    S.t.zero_()
    timed = S.advance(U.clone(), 2)
    ms, launches = S.kernel_timing(False)
    assert launches == 6 and ms > 0.0  # two steps of three stages, one axis
    assert torch.equal(plain, timed)
    S.close()
