"""The lane-parallel body step and force pass against the FP64 oracle, at the
sizes where their lane groups end: four lanes per body in 64-thread CTAs (16
bodies), eight in 128-thread CTAs (16 bodies), a warp per body for shapes of many
centres; one body per box (no force pass); and candidate lists that overflow.

Bodies stand in contact (inside the WCA cutoff) and three streaming steps are
compared, with the bars of the parity tests: |gpu - oracle| <= tol (|oracle| +
scale), tol 1e-12 (FP64 form) and 1e-5 (FP32 form: FP32 pair arithmetic), scale
the thermal value."""
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


def check(B, system, seed, steps=3):
    tol = TOL[system.params.precision]
    st = I.initial_state(system, seed)
    osys = O.OracleSystem(system)
    ost = O.OracleState(osys, st)
    sim = B.Simulation(system)
    sim.set_state(st)
    for _ in range(steps):
        sim.stream()
        O.stream(osys, ost)
    g = sim.get_state()
    sim.close()
    shp = system.body_shape_array()
    sP = np.sqrt([system.shapes[s].m.sum() for s in shp])[:, None]
    sL = np.sqrt([I.shape_inertia_diag(system.shapes[s]).max() for s in shp])[:, None]
    assert np.abs(g.R - ost.R).max() <= tol
    assert np.abs(g.q - ost.q).max() <= tol
    assert (np.abs(g.P - ost.P) / (np.abs(ost.P) + sP)).max() <= tol
    assert (np.abs(g.Lm - ost.Lm) / (np.abs(ost.Lm) + sL)).max() <= tol
    if system.n_bodies > system.n_rep:                # more than one in a box
        assert np.abs(ost.P - st.P).max() > 1e-3      # forces did act


def row(rng, n, gap, L):
    """n centres on a cubic lattice of spacing `gap`, jittered by 1 % of it"""
    k = int(L // gap)
    ijk = np.stack(np.unravel_index(np.arange(n), (k, k, k)), axis=1)
    return (ijk + 0.5) * gap + 0.01 * gap * rng.uniform(-1, 1, (n, 3))


@pytest.mark.parametrize("precision", [I.P64, I.P32])
@pytest.mark.parametrize("shape,n", [("sphere", 2), ("sphere", 15), ("sphere", 17), ("dumbbell", 16),
                                     ("dumbbell", 33), ("rod", 5)])
def test_bodies_in_contact(B, shape, n, precision):
    rng = np.random.default_rng(n)
    if shape == "sphere":
        sh, gap, L = I.sphere_shape(2.0, 1, 5.0), 4.05, 20
    elif shape == "dumbbell":
        sh, gap, L = I.dumbbell_shape(2.0, 0.2, 1, 5.0), 4.15, 20
    else:
        sh, gap, L = I.spherocylinder_shape(4.0, 6.0, 1.5, 5.0, cap_level=1), 6.02, 24
    R = row(rng, n, gap, L)
    q = I.random_quaternions(rng, n)
    if shape == "rod":
        q[:] = [1.0, 0.0, 0.0, 0.0]                   # end to end along z
    prm = I.Params(precision=precision, seed=n)
    check(B, I.build_system(prm, [sh], [(L, L, L)], 0.5, [[0] * n], "contact", R_q=[(R, q)]), n)


@pytest.mark.parametrize("precision", [I.P64, I.P32])
@pytest.mark.parametrize("n_rep", [1, 17])
def test_one_body_per_box(B, n_rep, precision):
    rng = np.random.default_rng(n_rep)
    sh = I.sphere_shape(2.0, 1, 5.0)
    R_q = [(rng.uniform(0, 10, (1, 3)), I.random_quaternions(rng, 1)) for _ in range(n_rep)]
    prm = I.Params(precision=precision, seed=3)
    check(B, I.build_system(prm, [sh], [(10, 10, 10)] * n_rep, 0.5, [[0]] * n_rep, "lone", R_q=R_q), 4)


@pytest.mark.parametrize("precision", [I.P64, I.P32])
def test_overflowing_candidate_lists(B, precision):
    rng = np.random.default_rng(9)
    small, big = I.sphere_shape(0.6, 0, 5.0), I.sphere_shape(3.0, 1, 5.0)
    R = row(rng, 360, 1.25, 15)                       # 10 by 12 by 3 of 12 by 12 by 12 places
    R = np.concatenate([R, [[7.5, 7.5, 11.0]]])
    q = I.random_quaternions(rng, len(R))
    prm = I.Params(precision=precision, seed=6)
    check(B, I.build_system(prm, [small, big], [(15, 15, 15)], 0.5, [[0] * 360 + [1]], "overflow", R_q=[(R, q)]), 5)


@pytest.mark.parametrize("precision", [I.P64, I.P32])
@pytest.mark.parametrize("sites", [3, 127, 128, 129, 256, 257, 640, 642, 768, 769, 1030])
def test_site_passes_at_their_edges(B, sites, precision):
    """One step with a shell of `sites` sites: the PRE and POST passes hold up to
    256 or 768 sites in registers and the rest in shared memory, in sums of 128
    lanes.  The bars are those of the parity tests (the site sums of the FP32 form
    are taken in FP32 by the device alone)."""
    rng = np.random.default_rng(sites)
    d = rng.standard_normal((sites, 3))
    b = 2.0 * d / np.linalg.norm(d, axis=1, keepdims=True)
    b -= b.mean(0)
    _, ax = np.linalg.eigh(b.T @ b)                   # principal axes
    sh = I.Shape(b=b @ ax, m=np.full(sites, 5.0), centres=np.zeros((1, 3)), wca_d=4.0)
    R = np.array([[3.0, 4.0, 5.0], [9.0, 10.0, 4.0]])
    prm = I.Params(precision=precision, thermostat=1, seed=sites)
    system = I.build_system(prm, [sh], [(13, 13, 13)], 5.0, [[0, 0]], "edges", R_q=[(R, I.random_quaternions(rng, 2))])
    st = I.initial_state(system, 1)
    osys = O.OracleSystem(system)
    ost = O.OracleState(osys, st)
    sim = B.Simulation(system)
    sim.set_debug(True)
    sim.set_state(st)
    sim.stream()
    O.stream(osys, ost)
    sim.couple(B.MPCD_PRE)
    sim.collide()
    dbg = sim.debug_cells()
    sim.couple(B.MPCD_POST)
    tr = O.collide(osys, ost)
    g = sim.get_state()
    sim.close()
    tol = TOL[precision]
    assert np.array_equal(dbg["site_cell"], tr["cell_site"])
    assert (np.abs(dbg["site_v"] - tr["site_v"]) / (np.abs(tr["site_v"]) + np.sqrt(1 / 5.0))).max() <= tol
    sP, sL = np.sqrt(sh.m.sum()), np.sqrt(I.shape_inertia_diag(sh).max())
    assert (np.abs(g.P - ost.P) / (np.abs(ost.P) + sP)).max() <= tol
    assert (np.abs(g.Lm - ost.Lm) / (np.abs(ost.Lm) + sL)).max() <= tol


@pytest.mark.parametrize("precision", [I.P64, I.P32])
@pytest.mark.parametrize("length", [5.0, 9.0, 13.0])
def test_rods_crossing_the_box(B, length, precision):
    """Rods in a box little longer than they are, packed at every angle and through
    its faces: the rows of centre pairs that are left out are those out of reach."""
    rng = np.random.default_rng(int(length))
    sh = I.spherocylinder_shape(2.4, length, 1.5, 5.0, cap_level=1)
    R, q, placed = I.rsa_place(rng, (14, 14, 14), [sh], [0] * 60, gap=0.0, max_attempts=300)
    prm = I.Params(precision=precision, seed=int(length))
    check(B, I.build_system(prm, [sh], [(14, 14, 14)], 0.5, [placed], "rods", R_q=[(R, q)]), 2)
