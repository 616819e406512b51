"""Bodies without a moment of inertia about some of their axes - one site: none at all;
sites in a row: none about the row - beside spheres.  The body step takes eight bodies
to a warp, so all kinds stand in one warp here, at counts around its eight, one body per
box and several: three streaming steps against the oracle with the bars of the parity
tests (|gpu - oracle| <= tol (|oracle| + scale), tol 1e-12 in the FP64 form and 1e-5 in
the FP32 form, scale the thermal value), and whole steps of the FP32 form bit for bit the
single calls."""
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


def shapes():
    out = [I.Shape(b=np.zeros((1, 3)), m=np.array([5.0]), centres=np.zeros((1, 3)), wca_d=1.5)]
    for axis in range(3):
        b = np.zeros((5, 3))
        b[:, axis] = np.linspace(-0.6, 0.6, 5)
        out.append(I.Shape(b=b, m=np.full(5, 5.0), centres=b[[0, 4]].copy(), wca_d=1.5))
    out.append(I.sphere_shape(0.8, 1, 5.0))
    for sh, zeros in zip(out, (3, 1, 1, 1, 0)):
        assert (I.shape_inertia_diag(sh) == 0.0).sum() == zeros
    return out


def box(n, lone, precision):
    rng = np.random.default_rng(n + 100 * lone)
    kinds = [int(k) for k in rng.permutation(np.arange(n) % 5)]
    q = I.random_quaternions(rng, n)
    if lone:
        L, R_q, per_box = (9, 9, 9), [(rng.uniform(0, 9, (1, 3)), q[i:i + 1]) for i in range(n)], [[k] for k in kinds]
    else:
        ijk = np.stack(np.unravel_index(np.arange(n), (6, 6, 6)), axis=1)
        R = (ijk + 0.5) * 2.6 + 0.1 * rng.uniform(-1, 1, (n, 3))     # near enough for forces
        L, R_q, per_box = (16, 16, 16), [(R, q)], [kinds]
    prm = I.Params(precision=precision, seed=n)
    system = I.build_system(prm, shapes(), [L] * len(per_box), 0.5, per_box, "moments", R_q=R_q)
    return system, I.initial_state(system, n)


@pytest.mark.parametrize("precision", [I.P64, I.P32])
@pytest.mark.parametrize("lone", [False, True])
@pytest.mark.parametrize("n", [2, 7, 8, 9, 19])
def test_streaming_against_the_oracle(B, n, lone, precision):
    tol = TOL[precision]
    system, st = box(n, lone, precision)
    osys = O.OracleSystem(system)
    ost = O.OracleState(osys, st)
    sim = B.Simulation(system)
    sim.set_state(st)
    for _ in range(3):
        sim.stream()
        O.stream(osys, ost)
    g = sim.get_state()
    sim.close()
    shp = system.body_shape_array()
    sP = np.sqrt([system.shapes[s].m.sum() for s in shp])[:, None]
    sL = np.sqrt([max(I.shape_inertia_diag(system.shapes[s]).max(), 1.0) for s in shp])[:, None]
    assert np.abs(g.R - ost.R).max() <= tol
    assert np.abs(g.q - ost.q).max() <= tol
    assert (np.abs(g.P - ost.P) / (np.abs(ost.P) + sP)).max() <= tol
    assert (np.abs(g.Lm - ost.Lm) / (np.abs(ost.Lm) + sL)).max() <= tol


@pytest.mark.parametrize("lone", [False, True])
@pytest.mark.parametrize("n", [8, 19])
def test_whole_steps_equal_single_calls(B, n, lone):
    system, st = box(n, lone, I.P32)
    a, b = B.Simulation(system), B.Simulation(system)
    for sim in (a, b):
        sim.set_state(st)
    a.step(3)
    for _ in range(3):
        b.stream()
        b.couple(B.MPCD_PRE)
        b.collide()
        b.couple(B.MPCD_POST)
    x, y = a.get_state(), b.get_state()
    for k in ("x", "v", "R", "q", "P", "Lm"):
        assert np.array_equal(getattr(x, k), getattr(y, k)), k
    a.close()
    b.close()
