"""The autograd function of the refinement on the host: what it does with the
library's results, with stand-ins on CPU tensors for the calls that need a GPU."""
import pytest

torch = pytest.importorskip("torch")

from paper_2006_01201_gb300 import binding, refine  # noqa: E402


@pytest.fixture
def quadratic(monkeypatch):
    """E(u) = sum u^2 (T0 and J0 do not matter) through the one-call entry
    points, which fill plain buffers and read `scale` through its pointer."""

    def energy(T0, J0, u, level, alpha):
        return (u.detach().double() ** 2).sum()

    def grad(T0, J0, u, level, alpha, scale=None, want_u=True, want_T=True, want_J=True):
        f = 1.0
        if scale is not None:
            scale.data_ptr()
            f = float(scale.detach())
        zero = torch.zeros_like(T0)
        return ((2 * f * u).detach() if want_u else None, zero if want_T else None, zero if want_J else None)

    monkeypatch.setattr(binding, "refine_energy", energy)
    monkeypatch.setattr(binding, "refine_grad", grad)
    g = torch.Generator().manual_seed(3)
    T, J = torch.rand((5, 7), generator=g), torch.rand((5, 7), generator=g)
    return T, J, torch.randn((5, 7, 2), generator=g)


def test_gradients_stay_differentiable_in_the_incoming_one(quadratic):
    T, J, u = quadratic
    v = torch.randn(u.shape, generator=torch.Generator().manual_seed(4))
    # jvp differentiates the gradient by the incoming one
    _, d = torch.autograd.functional.jvp(lambda x: refine.pyramid_energy(T, J, x), u, v)
    assert float(d) == pytest.approx(float((2 * u * v).double().sum()), rel=1e-5)
    x = u.clone().requires_grad_(True)
    g = torch.ones((), dtype=torch.float64, requires_grad=True)
    (du,) = torch.autograd.grad(refine.pyramid_energy(T, J, x), x, grad_outputs=g, create_graph=True)
    assert du.requires_grad
    (dg,) = torch.autograd.grad((du * v).sum(), g)
    assert float(dg) == pytest.approx(float((2 * u * v).double().sum()), rel=1e-5)


def test_a_batch_of_incoming_gradients(quadratic):
    T, J, u = quadratic
    x = u.clone().requires_grad_(True)
    g = torch.tensor([1.0, -2.5, 0.25], dtype=torch.float64)
    (du,) = torch.autograd.grad(refine.pyramid_energy(T, J, x), x, grad_outputs=g, is_grads_batched=True)
    torch.testing.assert_close(du, g.float()[:, None, None, None] * 2 * u)
    jac = torch.autograd.functional.jacobian(lambda y: refine.pyramid_energy(T, J, y), u, vectorize=True)
    torch.testing.assert_close(jac.float(), 2 * u)


@pytest.mark.parametrize("call", [lambda T, J, u: binding.energy_grad(T, J, u, 0.05),
                                  lambda T, J, u: binding.refine_energy(T, J, u, 0, 0.05),
                                  lambda T, J, u: binding.refine_grad(T, J, u, 0, 0.05)],
                         ids=["energy_grad", "refine_energy", "refine_grad"])
def test_planes_that_differ_are_refused(call):
    # before anything is read: the kernels use T's size for both planes
    T, u = torch.zeros((8, 6)), torch.zeros((8, 6, 2))
    for J in (torch.zeros((7, 6)), torch.zeros((8, 5)), torch.zeros((9, 6)), torch.zeros((8, 6), device="meta")):
        with pytest.raises(binding.PanoError, match="differ") as e:
            call(T, J, u)
        assert e.value.status == binding.PANO_ERR_INVALID_ARG


def test_planes_of_two_sizes_with_equal_levels(monkeypatch):
    # 100 and 99 rows are 50 at level 1: each plane's gradient has its own size
    down = lambda t: torch.zeros(((t.shape[0] + 1) // 2, (t.shape[1] + 1) // 2))
    monkeypatch.setattr(binding, "stage_pyr_down", down)

    def adjoint(g, h, w):
        assert tuple(g.shape) == ((h + 1) // 2, (w + 1) // 2)
        return torch.ones((h, w))

    monkeypatch.setattr(binding, "stage_pyr_down_adjoint", adjoint)
    monkeypatch.setattr(binding, "energy_grad", lambda T, J, u, alpha, **k: (
        torch.zeros((), dtype=torch.float64), torch.ones_like(u), torch.ones_like(T), torch.ones_like(J)))
    T0, J0 = torch.zeros((100, 40), requires_grad=True), torch.zeros((99, 39), requires_grad=True)
    u = torch.zeros((50, 20, 2), requires_grad=True)
    refine.pyramid_energy(T0, J0, u, 1).backward()
    assert T0.grad.shape == T0.shape and J0.grad.shape == J0.shape and u.grad.shape == u.shape


@pytest.mark.parametrize("level", [12, -1])
def test_levels_beyond_the_one_call_form(monkeypatch, quadratic, level):
    # pano_refine_* take levels 0 .. 11; the per-stage calls have no limit
    def refuse(*a, **k):
        raise binding.PanoError(binding.PANO_ERR_INVALID_ARG, "level not in 0..11")

    T, J, _ = quadratic
    monkeypatch.setattr(binding, "refine_energy", refuse)
    monkeypatch.setattr(binding, "refine_grad", refuse)
    monkeypatch.setattr(binding, "stage_pyr_down",
                        lambda t: torch.zeros(((t.shape[0] + 1) // 2, (t.shape[1] + 1) // 2)))
    monkeypatch.setattr(binding, "stage_pyr_down_adjoint", lambda g, h, w: torch.ones((h, w)))
    monkeypatch.setattr(binding, "energy_grad", lambda T, J, u, alpha, **k: (
        torch.zeros((), dtype=torch.float64), torch.ones_like(u), torch.ones_like(T), torch.ones_like(J)))
    T, u = T.clone().requires_grad_(True), torch.zeros((1, 1, 2), requires_grad=True)
    refine.pyramid_energy(T, J, u, level).backward()
    assert T.grad.shape == T.shape and u.grad.shape == u.shape


@pytest.mark.parametrize("plane", [torch.zeros((7, 1)).t(), torch.empty_strided((7, 1), (1, 7)), torch.zeros((1, 9))[:, ::3],
                                   torch.zeros((3, 1, 2))[:, :, 1], torch.zeros((6, 8))[:, 2:5]])
def test_strides_of_planes_at_level_0(monkeypatch, plane):
    # planes are made contiguous at level 0, whatever their strides; the stride
    # of a side of one element says nothing
    monkeypatch.setattr(torch.Tensor, "is_cuda", True, raising=False)
    h, w = plane.shape
    _, args, _ = binding._refine_args(plane, plane, torch.zeros((h, w, 2)), 0)
    assert args[2:7] == (h, w, w, w, 0)
