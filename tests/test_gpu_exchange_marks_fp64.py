"""The exchange's marks with the other arithmetic and rule: the FP64 form decides on doubles, and
MPCD-AT's binning draws and keeps normals beside the marks.  Whole steps (marked blocks only)
against the unpipelined calls (every particle): the same number of pairs and the same
state, bit for bit (FP32 form) or to the order of summation (1e-9 over seven steps, FP64 form)."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,rule", [(I.P64, I.SRD), (I.P64, I.AT), (I.P32, I.AT)])
@pytest.mark.parametrize("n", [1025, 9000])
@pytest.mark.parametrize("pairs,period,slabs", [(30, 1, (0.0, 7.0)), (1000, 3, (6.0, 0.0))])
def test_marked_scan_finds_the_same_pairs(n, pairs, period, slabs, precision, rule):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding as B, build_lib
    build_lib.build()
    prm = I.Params(rule=rule, thermostat=1, precision=precision, seed=n)
    system = I.System(prm, [I.sphere_shape(2.0, 0, 5.0)], [I.Replica(L=(8, 14, 9), n_solvent=n, body_shapes=[])])
    st = I.initial_state(system)

    def run(whole):
        sim = B.Simulation(system, sort_period=2 if whole else -1)
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
    assert na == nb and na > 0
    assert abs(pa - pb) <= 1e-9 * max(1.0, abs(pb))
    for k in ("x", "v"):
        u, w = getattr(a, k), getattr(b, k)
        if precision == I.P32:
            assert np.array_equal(u, w), k
        else:
            assert np.allclose(u, w, rtol=0.0, atol=1e-9 * max(1.0, np.abs(w).max())), k
