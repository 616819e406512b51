"""The solvent passes of the angular-momentum-conserving variants take each tile in
units of 256 particles: the state must not depend on how the tiles divide into them
(tiles below, at and just above a unit, ends of replicas inside a unit), bit for bit in
the FP32 form and to the order of summation (1e-12) in the FP64 form."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [I.P32, I.P64])
@pytest.mark.parametrize("rule", [I.SRD, I.AT])
def test_same_state_for_every_tile(rule, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding as B, build_lib
    build_lib.build()
    prm = I.Params(rule=rule, precision=precision, seed=6, angular=1)
    system = I.build_system(prm, [I.sphere_shape(1.5, 1, 5.0)], [(9, 8, 11), (5, 6, 5), (3, 3, 3)], 5.0,
                            [[0], [], []], "units",
                            R_q=[(np.array([[3.0, 4.0, 4.0]]), np.array([[1.0, 0.0, 0.0, 0.0]]))] +
                                [(np.zeros((0, 3)), np.zeros((0, 4)))] * 2)
    st = I.initial_state(system)

    def run(tile):
        sim = B.Simulation(system, sort_period=2)
        sim.set_tuning(block=128, tile=tile, ctas_per_sm=2, staged=0)
        sim.set_state(st)
        sim.step(4)
        g = sim.get_state()
        sim.close()
        return g

    ref = run(64)
    for tile in (128, 256, 264, 512, 1016):
        got = run(tile)
        for k in ("x", "v", "R", "q", "P", "Lm"):
            u, w = getattr(got, k), getattr(ref, k)
            if precision == I.P32:
                assert np.array_equal(u, w), (tile, k)
            else:
                assert np.allclose(u, w, rtol=0.0, atol=1e-12 * max(1.0, np.abs(w).max())), (tile, k)
