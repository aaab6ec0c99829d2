"""The FP32 filter's decisions at its range's edges are the FP64 ones: sides whose shock indicator
vanishes (eta -> 0, [beta] = 7, a clamp and not a threshold), and sides with one candidate on a flat
that carries nothing but rounding noise (its indicator may vanish)."""
import numpy as np
import pytest

from paper_2010_13289_gb300 import problems as PB

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,bc", [((64, 40), (0, 1)), ((33, 18, 17), (0, 0, 1))])
@pytest.mark.parametrize("amp", [1e-3, 0.3])
@pytest.mark.parametrize("noise", [1e-3, 0.0])
@pytest.mark.parametrize("K", [6, 8])
def test_filtered_decisions_on_flats(shape, bc, amp, noise, K):
    """Slopes that meet flats, with a perturbation of 1e-3 of the slope or of none but rounding
    (noise 0): decisions and C_T exponents are the FP64 ones, bit for bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2010_13289_gb300 import tenom as T
    prim = PB.random_state(tuple(reversed(shape)), 5, jumps=False)
    flat = np.zeros_like(prim)
    flat[0], flat[1], flat[-1] = 1.0, 0.3, 1.0
    ramp = np.zeros(prim.shape[1:])
    for a in range(ramp.ndim):   # slopes of every size that meet flats
        i = np.arange(ramp.shape[a])
        k = np.where(i % 8 < 4, i % 8, 4).astype(float) * (1 + i // 8 % 3)
        ramp += k.reshape([-1 if b == a else 1 for b in range(ramp.ndim)])
    prim = flat + amp * (0.05 * ramp + noise * (prim - prim.mean(axis=tuple(range(1, prim.ndim)), keepdims=True)))
    prim = torch.from_numpy(np.ascontiguousarray(prim)).cuda()
    dx = tuple(1.0 / n for n in shape)
    A = T.Solver(shape, dx, bc, T.make_scheme(K, limiter=0))
    B = T.Solver(shape, dx, bc, T.make_scheme(K, limiter=0, decisions=T.DECIDE_FP64))
    U = A.init_state(prim)
    for axis in range(len(shape)):
        d = T.stats_dict(A.decision_stats(U, axis).cpu(), K)
        assert d["certified_disagree"] == 0
        fa, fb = A.face_dump(U, axis, flags=True)[1], B.face_dump(U, axis, flags=True)[1]
        assert torch.equal(fa, fb)
    assert A.status() == 0 and B.status() == 0
    A.close()
    B.close()
