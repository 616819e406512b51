"""The +a solve forms its reciprocals from a coarse one where the argument is of moderate
size and by a division elsewhere.  The correction of given velocities does not depend on
the solvent's mass, and a power of two changes no rounding: the FP64 form must give the
same velocities for masses at which both paths are taken and the determinant (the cube of
the mass times up to 2^135) is a normal number.  Only the order of the sums of momenta
differs (1e-16 of them), which the solve of a nearly collinear cell enlarges:
1e-9 of the largest velocity, where a wrong reciprocal is off by more than all of it."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [-300, -200, 60, 200, 290])
def test_correction_does_not_depend_on_the_mass(power):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding as B, build_lib
    build_lib.build()

    def system(mass):
        prm = I.Params(rule=I.SRD, thermostat=0, precision=I.P64, seed=8, angular=1, m_solvent=mass)
        return I.build_system(prm, [I.sphere_shape(1.5, 1, 5.0)], [(6, 7, 5)], 8.0, [[]], "mass",
                              R_q=[(np.zeros((0, 3)), np.zeros((0, 4)))])

    st = I.initial_state(system(1.0))
    out = []
    for mass in (1.0, 2.0 ** power):
        sim = B.Simulation(system(mass))
        sim.set_state(st)
        sim.collide()
        out.append(np.array(sim.get_state().v))
        sim.close()
    assert not np.array_equal(out[0], np.asarray(st.v))
    assert np.abs(out[1] - out[0]).max() <= 1e-9 * np.abs(out[0]).max()
