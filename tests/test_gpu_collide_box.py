"""The one-launch collision (mpcd_collide_solvent_static) at the sizes where its
forms change: one cluster up to 32768 particles and 16384 cells, a cooperative
grid beyond, more than one group of four particles per thread beyond the resident
grid.  The same solvent in a context (mpcd_collide) must give the same velocities
bit for bit: integer sums, the same arithmetic per cell and particle."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding, build_lib
    build_lib.build()
    return binding, torch


def solvent(L, n, rule, thermostat, seed):
    prm = I.Params(rule=rule, thermostat=thermostat, precision=I.P32, seed=seed)
    system = I.System(prm, [I.sphere_shape(2.0, 0, 5.0)], [I.Replica(L=L, n_solvent=n, body_shapes=[])])
    return system, I.initial_state(system)


def gpu_rows(torch, a):
    return [torch.tensor(np.ascontiguousarray(a[:, k], dtype=np.float32), device="cuda") for k in range(3)]


@pytest.mark.parametrize("rule,thermostat", [(I.SRD, 0), (I.SRD, 1), (I.SRD, 2), (I.AT, 0)])
@pytest.mark.parametrize("L,n", [((3, 3, 3), 4), ((3, 4, 5), 36), ((17, 13, 19), 20992), ((20, 20, 20), 32768),
                                 ((20, 20, 20), 32772), ((25, 25, 26), 1004), ((32, 32, 16), 30000),
                                 ((40, 40, 40), 640000), ((20, 21, 19), 1300004)])
def test_matches_the_context(env, L, n, rule, thermostat):
    B, torch = env
    system, st = solvent(L, n, rule, thermostat, seed=n % 97 + 1)
    sim = B.Simulation(system, sort_period=-1)
    sim.set_state(st)
    sim.collide()
    want = sim.get_state().v
    sim.close()
    x, v = gpu_rows(torch, st.x), gpu_rows(torch, st.v)
    tag = torch.arange(n, dtype=torch.int32, device="cuda")
    for _ in range(2):                                # the scratch is left as it is found
        w = [t.clone() for t in v]
        B.collide_solvent_static(system.params, L, *x, *w, tag, step=0)
        got = np.stack([t.cpu().numpy() for t in w], axis=1)
        assert np.array_equal(got, want.astype(np.float32))


@pytest.mark.parametrize("L,n", [((12, 12, 12), 8640), ((40, 40, 40), 320000)])
def test_captured_in_a_graph(env, L, n):
    B, torch = env
    system, st = solvent(L, n, I.SRD, 1, seed=5)
    x, v = gpu_rows(torch, st.x), gpu_rows(torch, st.v)
    plain = [t.clone() for t in v]
    B.collide_solvent_static(system.params, L, *x, *plain, None, step=3)
    w = [t.clone() for t in v]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.collide_solvent_static(system.params, L, *x, *w, None, step=3)
    for _ in range(2):
        for a, b in zip(w, v):
            a.copy_(b)
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(w, plain))
