"""Bodies without solvent: a call of one step begins with the body step, right behind the
advance of the step counter, which the site PRE pass reads before it waits for the chain.
Many calls of one step, one call of all, and the single calls give the same state bit for
bit (FP32 form), one body per box and several."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("thermostat", [0, 1])
@pytest.mark.parametrize("per_box", [1, 3])
def test_same_state_however_the_steps_are_run(per_box, thermostat):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding as B, build_lib
    build_lib.build()
    rng = np.random.default_rng(per_box)
    prm = I.Params(thermostat=thermostat, precision=I.P32, seed=7)
    reps = [I.Replica(L=(14, 9, 9), n_solvent=0, body_shapes=[0] * per_box, id=i) for i in range(20)]
    system = I.System(prm, [I.sphere_shape(2.0, 2, 5.0)], reps)
    system._placements = [(np.array([[2.5, 4.0, 4.0], [7.0, 4.0, 4.5], [11.5, 4.5, 4.0]])[:per_box],
                           I.random_quaternions(rng, per_box)) for _ in reps]
    st = I.initial_state(system)

    def run(calls):
        sim = B.Simulation(system)
        sim.set_state(st)
        calls(sim)
        g = sim.get_state()
        sim.close()
        return g

    def ones(sim):
        for _ in range(60):
            sim.step(1)

    def singles(sim):
        for _ in range(60):
            sim.stream()
            sim.couple(B.MPCD_PRE)
            sim.collide()
            sim.couple(B.MPCD_POST)

    want = run(singles)
    assert np.isfinite(want.P).all() and not np.array_equal(want.P, st.P)
    for calls in (ones, lambda sim: sim.step(60)):
        got = run(calls)
        for k in ("R", "q", "P", "Lm"):
            assert np.array_equal(getattr(got, k), getattr(want, k)), k
