"""The FP32 screen of the face sweeps against FP64 decisions: a face the screen certifies
(its flux is the central one) must be one whose every candidate the FP64 cutoff keeps, so the
face fluxes of a scheme with filtered decisions equal those of the same scheme that decides
every face in FP64.  Sizes sit at the edges of the screen's tiles (64 faces in 1D, 256 along
x, 16 x 16 across) and at the shortest lines; states run from flat to broadband, subsonic and
supersonic, with stagnation points and jumps."""
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


def state(shape, kind, seed):
    prim = PB.random_state(tuple(reversed(shape)), seed, jumps=kind in ("jumps", "fast"))
    if kind == "faint":       # a small perturbation of a uniform stream
        base = np.zeros_like(prim)
        base[0], base[-1] = 1.0, 1.0
        prim = base + 1e-3 * (prim - prim.mean(axis=tuple(range(1, prim.ndim)), keepdims=True))
    elif kind == "fast":      # supersonic along every axis
        prim[1:-1] += 4.0
    elif kind == "flat":      # uniform but for one disturbed corner
        keep = prim[(slice(None),) + tuple(slice(0, max(1, n // 3)) for n in prim.shape[1:])].copy()
        prim[:] = np.array([1.0] + [0.0] * len(shape) + [0.7]).reshape((-1,) + (1,) * len(shape))
        prim[(slice(None),) + tuple(slice(0, n) for n in keep.shape[1:])] = keep
    return prim


CASES = [((4,), (0,), 8), ((3,), (1,), 6), ((63,), (1,), 6), ((64,), (0,), 8), ((129,), (1,), 8),
         ((16, 16), (0, 0), 6), ((257, 17), (0, 1), 8), ((255, 33), (1, 0), 6),
         ((17, 18, 15), (0, 0, 0), 8), ((16, 5, 33), (1, 0, 1), 6)]


@pytest.mark.parametrize("kind", ["smooth", "jumps", "faint", "fast", "flat"])
@pytest.mark.parametrize("shape,bc,K", CASES)
def test_screened_flux_equals_fp64_decisions(T, shape, bc, K, kind):
    """Tolerance: both evaluations round sums of at most about 100 terms of size max|F| of the
    component (the central sum, or projection, reconstruction and back-projection): 100 u =
    1e-14 typical, 1e-13 allowed; a wrongly certified face is off by its limiter's correction,
    which is of the order of the differences there (above 1e-6 in every state used)."""
    dx = tuple(1.0 / n for n in shape)
    prim = torch.from_numpy(np.ascontiguousarray(state(shape, kind, 3 + sum(shape) + K))).cuda()
    for lim in (0, 1):
        A = T.Solver(shape, dx, bc, T.make_scheme(K, limiter=lim))
        B = T.Solver(shape, dx, bc, T.make_scheme(K, limiter=lim, decisions=T.DECIDE_FP64))
        U = A.init_state(prim)
        for axis in range(len(shape)):
            Fa = A.face_dump(U, axis, flags=False)[0].cpu().numpy()
            Fb = B.face_dump(U, axis, flags=False)[0].cpu().numpy()
            big = np.abs(Fb).reshape(Fb.shape[0], -1).max(axis=1)
            # a component that vanishes analytically carries the rounding of the others
            big = np.maximum(big, 1e-2 * big.max())
            err = np.abs(Fa - Fb).reshape(Fb.shape[0], -1).max(axis=1)
            assert np.all(err <= 1e-13 * big), (axis, lim, err / big)
        assert A.status() == 0 and B.status() == 0
        A.close()
        B.close()
