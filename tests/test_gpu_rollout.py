"""Rollouts in one call per segment on lent scratch, against single steps on a
handle's own: states bit for bit, gradients to the rounding of the adjoint's
atomic sums; segments of one step, uneven, longer than the rollout; sizes whose
states end off a 16-byte boundary; the graph used twice and from another stream."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")
from paper_2509_08971_gb300 import autograd as AG  # noqa: E402


def _state(shape, dtype):
    g = torch.Generator(device="cuda").manual_seed(3)
    U = 0.1 * torch.rand((5,) + shape, generator=g, dtype=torch.float64, device="cuda")
    U[0] += 1.0
    U[4] += 2.5
    return U.to(dtype)


@pytest.mark.parametrize("shape", [(1, 1, 37), (1, 5, 7), (1, 33, 40), (3, 5, 9)])
@pytest.mark.parametrize("n,every", [(1, 1), (1, 4), (5, 1), (7, 3), (6, 3), (4, 9), (0, 3)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_rollout_equals_single_steps(shape, n, every, dtype):
    U0 = _state(shape, dtype)
    dts = [1e-3 * (1 + 0.1 * i) for i in range(n)]
    w = torch.randn(U0.shape, generator=torch.Generator(device="cuda").manual_seed(5), dtype=dtype,
                    device="cuda")
    m = hh.HardHydro(shape, 1.4, 0, dtype=dtype)
    states = [U0]
    for dt in dts:
        states.append(m.step(states[-1], dt))
    G, gg = w.clone(), torch.zeros((), dtype=torch.float64, device="cuda")
    for i in reversed(range(n)):
        G = m.step_backward(states[i], G, dts[i], gg)
    leaf = U0.clone().requires_grad_()
    gamma = torch.tensor(1.4, dtype=torch.float64, device="cuda", requires_grad=True)
    U = AG.rollout(leaf, gamma, AG.Mesh(shape, 0), dts, every)
    assert torch.equal(U, states[-1])
    tol = 1e-12 if dtype == torch.float64 else 1e-4
    for again in range(2):
        leaf.grad = gamma.grad = None
        with torch.no_grad():
            leaf.add_(0.0 if again == 0 else 1.0)        # the graph keeps its own first state
        (U * w).sum().backward(retain_graph=True)
        assert float((leaf.grad - G).abs().max()) <= tol * float(G.abs().max())
        assert abs(float(gamma.grad - gg)) <= tol * max(abs(float(gg)), 1.0)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        gU, = torch.autograd.grad(U, leaf, w)
    torch.cuda.synchronize()
    assert float((gU - G).abs().max()) <= tol * float(G.abs().max())


def test_lent_scratch():
    shape = (1, 12, 20)
    U = _state(shape, torch.float64)
    m = hh.HardHydro(shape, 1.4, 0, dtype=torch.float64)
    ref = m.step(U, 1e-3)                                # its own scratch first
    mem = m.workspace(0, U.device)
    assert torch.equal(m.step(U, 1e-3), ref) and m.get_error() == hh.HARD_OK
    n = hh.hard_hydro_workspace_bytes(m.h, 1)
    assert n > 0 and hh.hard_hydro_workspace_bytes(m.h, 2) == hh.HARD_EINVAL
    assert hh.hard_hydro_set_workspace(m.h, 0, mem.data_ptr(), 64, None) == hh.HARD_EINVAL
    assert hh.hard_hydro_set_workspace(m.h, 0, mem.data_ptr() + 4, mem.numel(), None) == hh.HARD_EINVAL
    assert hh.hard_hydro_steps(m.h, U.data_ptr(), [U.data_ptr()], [1e-3], None) == hh.HARD_EINVAL
    assert hh.hard_hydro_steps(m.h, U.data_ptr(), [ref.data_ptr()], [float("nan")], None) == hh.HARD_EINVAL
    # the other element type: the handle goes back to its own scratch
    assert hh.hard_hydro_set(m.h, hh.HARD_F32, 1.0, 1.0, 1.0, None) == hh.HARD_OK
    V = U.float()
    out = torch.empty_like(V)
    assert hh.hard_hydro_step(m.h, V.data_ptr(), out.data_ptr(), 1e-3, None) == hh.HARD_OK
    torch.cuda.synchronize()
    assert float((out - ref.float()).abs().max()) < 1e-5
