"""A caller's allocator need give no more than 16-byte alignment: the state after a
few steps is bit for bit that of the default allocator (FP32 form), or agrees to the
order of summation (FP64 form: 1e-12), from an allocator whose pointers are all 16
bytes past a 256-byte boundary."""
import numpy as np
import pytest

from paper_2604_14307_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("angular", [0, 1])
@pytest.mark.parametrize("precision", [I.P32, I.P64])
@pytest.mark.parametrize("rule", [I.SRD, I.AT])
def test_pointers_at_16_bytes(monkeypatch, rule, precision, angular):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_14307_gb300 import binding as B, build_lib
    build_lib.build()

    class Offset:
        def __init__(self, device):
            self._a = B.AllocFn(lambda n, _user: int(torch.cuda.caching_allocator_alloc(int(n) + 256, device)) + 16)
            self._f = B.FreeFn(lambda p, _user: torch.cuda.caching_allocator_delete(int(p) - 16))
            self.c = B.Allocator(self._a, self._f, None)

    prm = I.Params(rule=rule, precision=precision, seed=3, angular=angular)
    system = I.build_system(prm, [I.sphere_shape(1.5, 1, 5.0)], [(7, 9, 8), (5, 6, 5)], 5.0, [[0], []], "offset",
                            R_q=[(np.array([[3.0, 4.0, 4.0]]), np.array([[1.0, 0.0, 0.0, 0.0]])),
                                 (np.zeros((0, 3)), np.zeros((0, 4)))])
    st = I.initial_state(system)

    def run():
        sim = B.Simulation(system, sort_period=2)
        sim.set_state(st)
        sim.step(5)
        g = sim.get_state()
        sim.close()
        return g

    ref = run()
    monkeypatch.setattr(B, "_TorchAllocator", Offset)
    got = run()
    for k in ("x", "v", "R", "q", "P", "Lm"):
        u, w = getattr(got, k), getattr(ref, k)
        if precision == I.P32:
            assert np.array_equal(u, w), k
        else:
            assert np.allclose(u, w, rtol=0.0, atol=1e-12 * max(1.0, np.abs(w).max())), k
