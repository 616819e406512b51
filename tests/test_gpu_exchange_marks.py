"""The exchange inside whole steps reads only the blocks of slots that the solvent
pass marked.  Against the unpipelined calls, which read every particle: the same
pairs and the same state bit for bit (FP32 form), with slabs at block edges and
box faces, few and many pairs (candidates ranked or sorted), a period, re-sorts,
every launch form of the pass and the +a variant."""
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


@pytest.mark.parametrize("n", [5, 1023, 1025, 9000])
@pytest.mark.parametrize("pairs,period,slabs", [(1, 1, (0.0, 7.0)), (30, 2, (2.5, 13.0)), (1000, 3, (6.0, 0.0))])
@pytest.mark.parametrize("tuning,angular", [(None, 0), ((128, 256, 2, 1), 0), ((128, 256, 1, 2), 0),
                                            ((128, 256, 2, 0), 0), (None, 1)])
def test_marked_scan_finds_the_same_pairs(B, n, pairs, period, slabs, tuning, angular):
    prm = I.Params(thermostat=1, precision=I.P32, seed=n, angular=angular)
    system = I.System(prm, [I.sphere_shape(2.0, 0, 5.0)], [I.Replica(L=(8, 14, 9), n_solvent=n, body_shapes=[])])
    st = I.initial_state(system)

    def run(whole):
        sim = B.Simulation(system, sort_period=2 if whole else -1)
        if tuning:
            sim.set_tuning(block=tuning[0], tile=tuning[1], ctas_per_sm=tuning[2], staged=tuning[3])
        sim.set_state(st)
        sim.set_rnemd(y_a=slabs[0], y_b=slabs[1], max_pairs=pairs, period=period)
        if whole:
            sim.step(3)
            sim.step(4)
        else:
            for _ in range(7):
                sim.stream()
                sim.couple(B.MPCD_PRE)
                sim.collide()
                sim.couple(B.MPCD_POST)
        out = sim.get_state(), sim.rnemd_totals()
        sim.close()
        return out

    (a, (pa, na)), (b, (pb, nb)) = run(True), run(False)
    assert na == nb
    assert abs(pa - pb) <= 1e-12 * max(1.0, abs(pb))   # FP64 sums of the same terms, pair by pair
    assert np.array_equal(a.x, b.x) and np.array_equal(a.v, b.v)
