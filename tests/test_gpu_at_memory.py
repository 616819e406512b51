"""MPCD-AT asks for no more device memory than its cell words need: the normals of the solvent
lie in the solvent buffer that is not in use, and the normals of the sites are kept only
where there is memory for them.  The requests of a context against those of the SRD
rule for the same system; a context whose last request is refused, and one that has to give
the kept normals back for a protocol's buffers, take the same steps bit for bit (FP32 form)
or to the order of summation (1e-9, FP64 form)."""
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


def box(rule, precision, angular=0):
    prm = I.Params(rule=rule, precision=precision, seed=5, angular=angular)
    system = I.build_system(prm, [I.sphere_shape(1.5, 2, 5.0)], [(9, 8, 11), (5, 6, 5)], 5.0, [[0, 0], []], "memory",
                            R_q=[(np.array([[3.0, 4.0, 3.0], [6.0, 4.0, 8.0]]), np.array([[1.0, 0, 0, 0]] * 2)),
                                 (np.zeros((0, 3)), np.zeros((0, 4)))])
    return system, I.initial_state(system)


def allocator(env, budget=None):
    """A stand-in for the binding's allocator with a budget; its requests and what is held."""
    B, torch = env
    log = dict(requests=[], held={}, refused=0)

    class Budget:
        def __init__(self, device):
            def alloc(n, _user):
                n = int(n)
                if budget is not None and sum(log["held"].values()) + n > budget:
                    log["refused"] += 1
                    return None
                p = int(torch.cuda.caching_allocator_alloc(n, device))
                log["requests"].append(n)
                log["held"][p] = n
                return p

            def free(p, _user):
                log["held"].pop(int(p))
                torch.cuda.caching_allocator_delete(int(p))
            self._a, self._f = B.AllocFn(alloc), B.FreeFn(free)
            self.c = B.Allocator(self._a, self._f, None)
    return Budget, log


def up(n):
    return (n + 255) & ~255


def steps(env, monkeypatch, system, st, budget=None, lags=0):
    B, _ = env
    cls, log = allocator(env, budget)
    monkeypatch.setattr(B, "_TorchAllocator", cls)
    sim = B.Simulation(system, sort_period=2)
    at_start = sum(log["held"].values())
    sim.set_state(st)
    sim.step(2)
    if lags:
        sim.set_vacf(lags)
    sim.step(4)
    sim.stream()
    sim.couple(B.MPCD_PRE)
    sim.collide()
    sim.couple(B.MPCD_POST)
    g = sim.get_state()
    at_end = sum(log["held"].values())
    sim.close()
    assert not log["held"]                            # everything was given back
    return g, log, at_start, at_end


def agree(precision, a, b):
    for k in ("x", "v", "R", "q", "P", "Lm"):
        u, w = getattr(a, k), getattr(b, k)
        if precision == I.P32:
            assert np.array_equal(u, w), k
        else:
            assert np.allclose(u, w, rtol=0.0, atol=1e-9 * max(1.0, np.abs(w).max())), k


@pytest.mark.parametrize("precision", [I.P32, I.P64])
def test_requests(env, monkeypatch, precision):
    real = 4 if precision == I.P32 else 8
    system, st = box(I.AT, precision)
    cells, sites = sum(int(np.prod(r.L)) for r in system.replicas), system.n_sites
    _, _, at, _ = steps(env, monkeypatch, system, st)
    _, _, srd, _ = steps(env, monkeypatch, *box(I.SRD, precision))
    words = (4, 6) if precision == I.P32 else (6, 8)
    extra = up(cells * words[1] * 8) - up(cells * words[0] * 8)
    kept = up(3 * sites * real)
    assert at - srd <= extra + kept                   # (the tile tables follow the launch form)


@pytest.mark.parametrize("angular", [0, 1])
@pytest.mark.parametrize("precision", [I.P32, I.P64])
def test_without_the_sites_normals(env, monkeypatch, precision, angular):
    system, st = box(I.AT, precision, angular)
    want, _, total, _ = steps(env, monkeypatch, system, st)
    got, log, held, _ = steps(env, monkeypatch, system, st, budget=total - 1)
    assert log["refused"] == 1 and held < total
    agree(precision, got, want)


@pytest.mark.parametrize("precision", [I.P32, I.P64])
def test_given_back_for_a_protocol(env, monkeypatch, precision):
    system, st = box(I.AT, precision)
    want, _, total, end = steps(env, monkeypatch, system, st, lags=10)
    assert end > total
    got, log, held, after = steps(env, monkeypatch, system, st, budget=end - 1, lags=10)
    assert held == total and log["refused"] == 1 and after < end
    agree(precision, got, want)
