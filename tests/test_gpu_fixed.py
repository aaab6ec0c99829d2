"""The nonlinear faces' limiter corrections in 64-bit fixed point: face fluxes and cutoff flags
against the CPU oracle for the extremes that the form accepts (coefficients at the ends of
their range, both curvatures, values at and beyond the exponents where it hands over to FP64),
to the parity rules' 1e-13."""
import numpy as np
import pytest

from paper_2010_13289_gb300 import problems as PB
from parity import bound_counts, central_terms, compare_faces

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


CASES = [(6, 0, {}), (8, 0, {}), (6, 1, {}), (8, 1, {}), (6, 0, {"mp_alpha": 0.0, "mp_beta": 0.0}),
         (8, 0, {"mp_alpha": 7.9, "mp_beta": 23.9}), (8, 0, {"mp_alpha": 8.0}), (6, 0, {"mp_beta": 24.0}),
         (6, 0, {"mp_curv": 1, "mp_beta": 1.0})]


@pytest.mark.parametrize("scale", [1.0, 3e-10, 1e-13, 5e11, 1e14])
@pytest.mark.parametrize("K,lim,kw", CASES)
def test_fixed_point_corrections_match_oracle(T, orc, K, lim, kw, scale):
    """scale multiplies density and pressure (the velocities stay), hence every sequence."""
    shape, bc = (37, 29), (0, 0)  # (a zero-gradient ghost stencil overflows gamma at the large scales)
    prim = PB.random_state(tuple(reversed(shape)), seed=7 * K + lim, jumps=True)
    prim[0] *= scale
    prim[-1] *= scale
    dx = tuple(1.0 / n for n in shape)
    S = T.Solver(shape, dx, bc, T.make_scheme(K, limiter=lim, **kw))
    g, so = orc.make_grid(shape, dx, bc), orc.make_scheme(K, limiter=lim, **kw)
    Uo = orc.init_state(g, prim)
    Ug = torch.from_numpy(Uo).cuda()
    for a in range(2):
        Fg, flg = S.face_dump(Ug, a)
        Fo, flo, cut, noise, bad, sc = orc.faces(g, so, Uo, a, with_scale=True)
        sc = np.maximum(sc, central_terms(Uo, a, K, bc[a]))
        assert bad == 0
        st = compare_faces(Fg.cpu().numpy(), flg.cpu().numpy(), Fo, flo, cut, noise, sc,
                           label="fixed %s %g axis %d" % ((K, lim), scale, a))
        bound_counts(st, noise_frac=0.05)
    assert S.status() == 0
    S.close()
