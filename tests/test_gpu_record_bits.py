"""A recorded step is the step: tenom_rk3_step and the record calls write the same bits (a rollout is
recomputed from its checkpoints for the reverse, with the branches of the recomputed states)."""
import numpy as np
import pytest

from paper_2010_13289_gb300 import problems as PB

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [((9,), (1,)), ((500,), (1,)), ((1901,), (0,)), ((3000,), (0,)), ((100, 37), (0, 1)), ((30, 11, 17), (0, 1, 0))]


@pytest.mark.parametrize("shape,bc", SHAPES)
@pytest.mark.parametrize("K", [6, 8])
@pytest.mark.parametrize("lim", [0, 1])
def test_recorded_steps_have_the_bits_of_steps(shape, bc, K, lim):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2010_13289_gb300 import tenom as T
    prim = PB.random_state(tuple(reversed(shape)), K + lim, jumps=True)
    S = T.Solver(shape, tuple(1.0 / n for n in shape), bc, T.make_scheme(K, limiter=lim))
    U = S.init_state(torch.from_numpy(np.ascontiguousarray(prim)).cuda())
    dt = S.max_dt(U, 0.4).clone()
    plain = S.rk3_step(U.clone(), dt)
    for linear in (False, True):
        assert torch.equal(S.rk3_step_record(U.clone(), dt, S.new_tape(linear=linear)), plain), linear
    assert torch.equal(S.rhs_record(U, S.new_lin()), S.rhs(U))
    assert S.status() == 0
    S.close()
