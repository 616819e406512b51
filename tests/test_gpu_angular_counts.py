"""The +a variants in a cell of very many members: the counts of a cell are those of the
plain words (up to 65535 solvent particles and as many sites), and its words are
cleared whatever the counts are.

A small body lies with all its sites in one cell, at counts around multiples of 1024, and
a crowded box holds more than 4096 solvent particles a cell.  One collision against the
oracle, |gpu - oracle| <= bar (|oracle| + 1 + |w_c|): the FP64 bar is 1e-12 times the
square root of the sites (order of summation), the FP32 bar 1e-5 and 2^-20 a member (the
unit to which each member's momentum term is rounded).  And nothing of one step is left
for the next: a state read after every step and loaded into a new context goes on as the
steps do, bit for bit (FP32 form), to the order of summation (1e-9, FP64 form)."""
import numpy as np
import pytest

import oracle as O
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


def cluster(sites):
    d = np.random.default_rng(sites).standard_normal((sites, 3))
    b = 0.02 * d / np.linalg.norm(d, axis=1, keepdims=True)
    b -= b.mean(0)
    _, ax = np.linalg.eigh(b.T @ b)                   # principal axes
    return I.Shape(b=b @ ax, m=np.full(sites, 5.0), centres=np.zeros((1, 3)), wca_d=2.0)


def box(sites, rule, precision, density=5.0):
    prm = I.Params(rule=rule, thermostat=1, precision=precision, seed=1026, angular=1)
    L = (5, 6, 7)
    R = np.array([[2.3, 3.1, 3.6]])
    system = I.build_system(prm, [cluster(max(sites, 4))], [L], density, [[0] if sites else []], "cluster",
                            R_q=[(R, np.array([[1.0, 0.0, 0.0, 0.0]])) if sites else
                                 (np.zeros((0, 3)), np.zeros((0, 4)))])
    return system, I.initial_state(system)


def one_collision(B, system, st, members):
    sim = B.Simulation(system)
    sim.set_state(st)
    sim.step(1)
    g = sim.get_state()
    sim.close()
    osys = O.OracleSystem(system)
    ost = O.OracleState(osys, st)
    O.stream(osys, ost)
    tr = O.collide(osys, ost)
    p32 = system.params.precision == I.P32
    bar = 1e-5 + members * 2.0 ** -20 if p32 else 1e-12 * np.sqrt(max(members, 1))
    w = np.linalg.norm(tr["cell_omega"], axis=1)[tr["cell_solvent"]]
    assert (np.abs(g.v - ost.v) / (np.abs(ost.v) + 1.0 + w[:, None])).max() <= bar
    if system.n_bodies:
        wb = np.linalg.norm(tr["cell_omega"], axis=1)[tr["cell_site"]].max()
        m = system.shapes[0].m.sum()
        assert np.abs(g.P - ost.P).max() <= bar * (np.abs(ost.P).max() + m * (1.0 + wb))
    return tr


@pytest.mark.parametrize("precision", [I.P32, I.P64])
@pytest.mark.parametrize("rule", [I.SRD, I.AT])
@pytest.mark.parametrize("sites", [1023, 1024, 1025, 2048])
def test_all_sites_in_one_cell(B, sites, rule, precision):
    system, st = box(sites, rule, precision)
    tr = one_collision(B, system, st, sites)
    assert len(np.unique(tr["cell_site"])) == 1


@pytest.mark.parametrize("precision", [I.P32, I.P64])
def test_crowded_cells(B, precision):
    system, st = box(0, I.SRD, precision, density=4700.0)
    tr = one_collision(B, system, st, 4700)
    assert (np.bincount(tr["cell_solvent"]) >= 4096).all()


@pytest.mark.parametrize("precision", [I.P32, I.P64])
@pytest.mark.parametrize("rule", [I.SRD, I.AT])
def test_nothing_is_left_for_the_next_step(B, rule, precision):
    system, st = box(1024, rule, precision)
    a = B.Simulation(system)
    a.set_state(st)
    for _ in range(4):
        before = a.get_state()
        a.step(1)
        b = B.Simulation(system)
        b.set_state(before)
        b.step(1)
        x, y = a.get_state(), b.get_state()
        b.close()
        for k in ("x", "v", "R", "q", "P", "Lm"):
            u, w = getattr(x, k), getattr(y, k)
            if precision == I.P32:
                assert np.array_equal(u, w), k
            else:
                assert np.allclose(u, w, rtol=0.0, atol=1e-9 * max(1.0, np.abs(w).max())), k
    a.close()
