"""The FP64 form's cell parameters where their code changes course, against the
oracle: sums of up to 16 exponentials per logarithm (cells of 2 to 80 members,
odd and even numbers of degrees of freedom), the rejection sampler's squeeze, the
wrap at the box faces.  Bar of the FP64 parity tests: |gpu - oracle| <= 1e-12
(|oracle| + 1); positions bit for bit."""
import numpy as np
import pytest

import oracle as O
from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("thermostat", [1, 2])
@pytest.mark.parametrize("density", [0.7, 4.0, 11.3, 22.0, 60.0])
def test_cells_of_every_occupation(density, thermostat):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding, build_lib
    build_lib.build()
    L = (7, 9, 8)
    prm = I.Params(thermostat=thermostat, precision=I.P64, seed=int(10 * density))
    n = int(density * np.prod(L))
    system = I.System(prm, [I.sphere_shape(2.0, 0, 5.0)], [I.Replica(L=L, n_solvent=n, body_shapes=[])])
    st = I.initial_state(system)
    st.x[:6] = [[0.0, 0.0, 0.0], [6.999999999999999, 8.999999999999998, 7.999999999999999], [0.0, 4.0, 7.5],
                [1e-300, 1e-17, 2.0], [3.0, 0.0, 1e-18], [6.5, 8.5, 7.5]]
    st.v[:6] = [[-0.0, -1e-18, -1e-17], [1e-14, 1e-15, 1e-14], [-1e-20, 1.0, 5.0], [-1e-300, -1e-16, 0.0],
                [0.0, -0.0, -1e-17], [5.0, 5.0, 5.0]]
    sim = binding.Simulation(system)
    sim.set_state(st)
    sim.stream()
    sim.couple(binding.MPCD_PRE)
    sim.collide()
    sim.couple(binding.MPCD_POST)
    g = sim.get_state()
    sim.close()
    osys = O.OracleSystem(system)
    ost = O.OracleState(osys, st)
    O.step(osys, ost, 1)
    assert np.array_equal(g.x, ost.x)
    assert (np.abs(g.v - ost.v) / (np.abs(ost.v) + 1.0)).max() <= 1e-12
