"""Shapes whose thermal draws wait in shared memory (more than 768 sites).  The site PRE pass
takes 12 (FP32 form) or 24 bytes (FP64 form) a site beside its static arrays, so the counts
here stand around 48 KB without and with those of either form of the pass, and near all
that a CTA can have, where the form of two lanes per sum has no room.  Then the one-lane
form (more than eight bodies an SM) at the counts where the draws change place, and a
context of many sites that steps on after one of fewer was made.

One step against the oracle with the bars of the parity tests: |gpu - oracle| <= tol
(|oracle| + scale), tol 1e-12 (FP64 form) and 1e-5 (FP32 form), scale the thermal value."""
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


def shell(sites, radius=2.0):
    d = np.random.default_rng(sites).standard_normal((sites, 3))
    b = radius * d / np.linalg.norm(d, axis=1, keepdims=True)
    b -= b.mean(0)
    _, ax = np.linalg.eigh(b.T @ b)                   # principal axes
    return I.Shape(b=b @ ax, m=np.full(sites, 5.0), centres=np.zeros((1, 3)), wca_d=2 * radius)


def boxes(sites, precision, n_rep=1, per_box=2):
    rng = np.random.default_rng(sites)
    R = np.array([[3.0, 4.0, 5.0], [9.0, 10.0, 4.0]])[:per_box]
    prm = I.Params(precision=precision, thermostat=1, seed=sites)
    L = (13, 13, 13) if per_box > 1 else (6, 6, 6)
    system = I.build_system(prm, [shell(sites, 2.0 if per_box > 1 else 1.0)], [L] * n_rep, 1.0,
                            [[0] * per_box] * n_rep, "sites",
                            R_q=[(R, I.random_quaternions(rng, per_box)) for _ in range(n_rep)])
    return system, I.initial_state(system, 1)


def one_step(B, system, st):
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
    tol, sh = TOL[system.params.precision], system.shapes[0]
    assert np.array_equal(dbg["site_cell"], tr["cell_site"])
    assert (np.abs(dbg["site_v"] - tr["site_v"]) / (np.abs(tr["site_v"]) + np.sqrt(1 / 5.0))).max() <= tol
    sP, sL = np.sqrt(sh.m.sum()), np.sqrt(I.shape_inertia_diag(sh).max())
    assert (np.abs(g.P - ost.P) / (np.abs(ost.P) + sP)).max() <= tol
    assert (np.abs(g.Lm - ost.Lm) / (np.abs(ost.Lm) + sL)).max() <= tol


@pytest.mark.parametrize("precision,sites", [(I.P64, n) for n in (1774, 1775, 2004, 2014, 2015, 2048, 2049, 9412, 9413, 9600)] +
                         [(I.P32, n) for n in (3821, 3822, 4029, 4030, 4096, 4097, 19096, 19097, 19300)])
def test_draws_in_shared_memory(B, precision, sites):
    one_step(B, *boxes(sites, precision))


@pytest.mark.parametrize("precision", [I.P64, I.P32])
@pytest.mark.parametrize("sites", [256, 257, 768, 769])
def test_one_lane_per_sum(B, sites, precision):
    one_step(B, *boxes(sites, precision, n_rep=1230, per_box=1))


@pytest.mark.parametrize("precision,many,few", [(I.P64, 9000, 2100), (I.P32, 19000, 4200)])
def test_a_later_context_of_fewer_sites(B, precision, many, few):
    system, st = boxes(many, precision)
    a = B.Simulation(system)
    other = B.Simulation(boxes(few, precision)[0])
    a.set_state(st)
    a.step(2)
    assert np.isfinite(a.get_state().P).all()
    other.close()
    a.close()


def test_mixed_shapes_fp64(B):
    """The ensemble of spheres, dumbbells and rods (up to 2004 sites) in the FP64 form: whole
    steps agree with the single calls to the order of summation (1e-9)."""
    system = I.batched_mixed_shapes(3, seed=5, precision=I.P64)
    assert max(s.n_sites for s in system.shapes) > 1775
    st = I.initial_state(system)
    a, b = B.Simulation(system), B.Simulation(system)
    for sim in (a, b):
        sim.set_state(st)
    a.step(2)
    for _ in range(2):
        b.stream()
        b.couple(B.MPCD_PRE)
        b.collide()
        b.couple(B.MPCD_POST)
    x, y = a.get_state(), b.get_state()
    for k in ("x", "v", "R", "q", "P", "Lm"):
        u, w = getattr(x, k), getattr(y, k)
        assert np.allclose(u, w, rtol=0.0, atol=1e-9 * max(1.0, np.abs(w).max())), k
    a.close()
    b.close()
