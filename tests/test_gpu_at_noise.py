"""MPCD-AT keeps the normals of a binning for the collision that it is for.  They
must be drawn again wherever the storage order or the step has moved in between:
whole steps with re-sorts at every phase, explicit sorts between the calls, a
restored state.  Every way of running the same steps gives the same state bit for
bit (FP32 form), for every launch form of the pass and with a colloid."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding, build_lib
    build_lib.build()
    return binding


def same(a, b):
    return all(np.array_equal(getattr(a, k), getattr(b, k)) for k in ("x", "v", "R", "q", "P", "Lm"))


@pytest.mark.parametrize("tuning", [None, (128, 256, 2, 1), (128, 256, 1, 2), (64, 128, 1, 3), (128, 256, 2, 0)])
@pytest.mark.parametrize("angular", [0, 1])
def test_same_state_however_the_steps_are_run(B, angular, tuning):
    prm = I.Params(rule=I.AT, precision=I.P32, seed=4, angular=angular)
    system = I.build_system(prm, [I.sphere_shape(1.5, 1, 5.0)], [(7, 9, 8), (5, 6, 5)], 5.0, [[0], []], "noise",
                            R_q=[(np.array([[3.0, 4.0, 4.0]]), np.array([[1.0, 0.0, 0.0, 0.0]])),
                                 (np.zeros((0, 3)), np.zeros((0, 4)))])
    st = I.initial_state(system)

    def run(period, calls):
        sim = B.Simulation(system, sort_period=period)
        if tuning:
            sim.set_tuning(block=tuning[0], tile=tuning[1], ctas_per_sm=tuning[2], staged=tuning[3])
        sim.set_state(st)
        calls(sim)
        g = sim.get_state()
        sim.close()
        return g

    def singles(sim):
        for k in range(7):
            sim.stream()
            sim.couple(B.MPCD_PRE)
            sim.collide()
            if k % 2:
                sim.sort()
            sim.couple(B.MPCD_POST)

    def pieces(sim):
        for n in (1, 3, 2, 1):
            sim.step(n)

    def restored(sim):
        sim.step(3)
        sim.set_state(st)
        sim.step(7)

    want = run(-1, singles)
    assert same(want, run(1, lambda sim: sim.step(7)))
    assert same(want, run(2, pieces))
    assert same(want, run(3, pieces))
    assert same(want, run(20, restored))
