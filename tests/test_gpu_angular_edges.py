"""The +a variants' passes at the edges of their warps (128 particles a round, four
per lane, runs of equal cells that end anywhere): the oracle within the +a bar
|gpu - oracle| <= tol (|oracle| + 1 + |w_c|), w_c the cell's correction, tol 1e-5
(FP32 form) and 1e-12 (FP64 form); and whole steps (rule, solve, correction with
the next step's streaming and binning) bit for bit the single calls in the FP32
form, with and without a colloid, across a re-sort."""
import numpy as np
import pytest

import oracle as O
from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = {I.P64: 1e-12, I.P32: 1e-5}


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding, build_lib
    build_lib.build()
    return binding


def box(n, rule, precision, colloid=False):
    prm = I.Params(rule=rule, thermostat=1, precision=precision, seed=n + 1, angular=1)
    sh = I.sphere_shape(1.5, 1, 5.0)
    rep = I.Replica(L=(5, 6, 7), n_solvent=n, body_shapes=[0] if colloid else [])
    system = I.System(prm, [sh], [rep])
    if colloid:
        system._placements = [(np.array([[2.5, 3.0, 3.5]]), np.array([[1.0, 0.0, 0.0, 0.0]]))]
    return system, I.initial_state(system)


@pytest.mark.parametrize("precision", [I.P32, I.P64])
@pytest.mark.parametrize("rule", [I.SRD, I.AT])
@pytest.mark.parametrize("n", [1, 3, 127, 128, 129, 1023, 2051])
def test_one_collision(B, n, rule, precision):
    system, st = box(n, rule, precision)
    sim = B.Simulation(system)
    sim.set_state(st)
    sim.step(1)
    g = sim.get_state()
    sim.close()
    osys = O.OracleSystem(system)
    ost = O.OracleState(osys, st)
    O.stream(osys, ost)
    tr = O.collide(osys, ost)
    w = np.linalg.norm(tr["cell_omega"], axis=1)[tr["cell_solvent"]]
    assert np.array_equal(g.x, ost.x)
    assert (np.abs(g.v - ost.v) / (np.abs(ost.v) + 1.0 + w[:, None])).max() <= TOL[precision]


@pytest.mark.parametrize("colloid", [False, True])
@pytest.mark.parametrize("rule", [I.SRD, I.AT])
@pytest.mark.parametrize("n", [129, 1023, 2100])
def test_whole_steps_equal_single_calls(B, n, rule, colloid):
    system, st = box(n, rule, I.P32, colloid)
    a, b = B.Simulation(system, sort_period=2), B.Simulation(system, sort_period=-1)
    for sim in (a, b):
        sim.set_state(st)
    a.step(4)
    a.step(2)
    for _ in range(6):
        b.stream()
        b.couple(B.MPCD_PRE)
        b.collide()
        b.couple(B.MPCD_POST)
    x, y = a.get_state(), b.get_state()
    for k in ("x", "v", "R", "q", "P", "Lm"):
        assert np.array_equal(getattr(x, k), getattr(y, k)), k
    a.close()
    b.close()
