"""Differentiable refinement on the GPU against the FP64 oracle: energy and
gradients on a 64x64 crop of the 1024x1024 pair, central finite differences
of the GPU's FP64 energy, the REDUCE transpose, gradients through pyramid
levels, and refinement by gradient steps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synth  # noqa: E402

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2006_01201_gb300 import binding  # noqa: E402
from paper_2006_01201_gb300 import build as gpu_build  # noqa: E402
from paper_2006_01201_gb300 import refine  # noqa: E402

DEV = torch.device("cuda:0")
ALPHA = 0.05


@pytest.fixture(scope="module", autouse=True)
def _lib():
    gpu_build.build()
    binding.load_library()


@pytest.fixture(scope="module")
def pair1024():
    return synth.pair_small_gray(seed=3, h=1024, w=1024, amp_x=6.0, amp_y=3.0, levels=5)


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)


def crop(pair, y0=480, x0=480, n=64):
    T = pair.L[y0:y0 + n, x0:x0 + n].astype(np.float32)
    J = pair.R[y0:y0 + n, x0:x0 + n].astype(np.float32)
    u = pair.flow_LtoR[y0:y0 + n, x0:x0 + n].astype(np.float32)
    u = u + np.random.default_rng(4).normal(0, 0.3, u.shape).astype(np.float32)
    return T, J, u


def test_energy_and_gradients_match_oracle_on_crop(pair1024):
    T, J, u = crop(pair1024)
    E, gu, gt, gj = binding.energy_grad(cuda(T), cuda(J), cuda(u), ALPHA)
    torch.cuda.synchronize()
    Eo = oracle.energy(T, J, u, ALPHA)
    guo, gto, gjo = oracle.energy_grad(T, J, u, ALPHA)
    assert float(E) == pytest.approx(Eo, rel=1e-5)
    for got, ref in ((gu, guo), (gt, gto), (gj, gjo)):
        got = got.cpu().numpy()
        assert np.abs(got - ref).max() <= 1e-5 * max(1.0, np.abs(ref).max())


def test_gpu_gradient_matches_central_differences(pair1024):
    T, J, u = crop(pair1024)
    Tt, Jt, ut = cuda(T), cuda(J), cuda(u)
    _, gu, _, _ = binding.energy_grad(Tt, Jt, ut, ALPHA)
    g = np.random.default_rng(5)
    h = 1e-3
    for trial in range(6):
        # every coordinate moves by h (random signs): smaller per-pixel steps
        # would drown in the FP32 rounding of the residuals
        d = g.choice([-1.0, 1.0], size=u.shape).astype(np.float32)
        if trial >= 3:                      # single coordinates as well
            d = np.zeros_like(u)
            d[g.integers(0, 64), g.integers(0, 64), g.integers(0, 2)] = 1.0
        dt = cuda(d)
        Ep = float(binding.energy_grad(Tt, Jt, ut + h * dt, ALPHA, want_u=False, want_T=False, want_J=False)[0])
        Em = float(binding.energy_grad(Tt, Jt, ut - h * dt, ALPHA, want_u=False, want_T=False, want_J=False)[0])
        fd = (Ep - Em) / (2 * h)
        an = float((gu.double() * dt.double()).sum())
        assert abs(fd - an) <= 2e-3 * max(abs(an), 1e-2), (trial, fd, an)


@pytest.mark.parametrize("shape", [(37, 53), (64, 64), (5, 2), (1, 9)])
def test_reduce_transpose_on_gpu(shape):
    g = np.random.default_rng(6)
    x = g.normal(size=shape).astype(np.float32)
    y = g.normal(size=((shape[0] + 1) // 2, (shape[1] + 1) // 2)).astype(np.float32)
    Ax = binding.stage_pyr_down(cuda(x)).cpu().numpy().astype(np.float64)
    ATy = binding.stage_pyr_down_adjoint(cuda(y), *shape).cpu().numpy().astype(np.float64)
    lhs, rhs = float((Ax * y).sum()), float((x * ATy).sum())
    assert lhs == pytest.approx(rhs, rel=1e-5, abs=1e-5)
    np.testing.assert_allclose(ATy, oracle.pyr_down_adjoint(y, *shape), rtol=0, atol=1e-6)


def test_pyramid_energy_gradients_through_levels():
    p = synth.pair_small_gray(seed=7, h=96, w=128, amp_x=2.0, amp_y=1.0, levels=3)
    level = 2
    T0, J0 = cuda(p.L), cuda(p.R)
    pyrT = oracle.pyramid(p.L, level + 1)
    pyrJ = oracle.pyramid(p.R, level + 1)
    hl, wl = pyrT[level].shape
    u = np.random.default_rng(8).normal(0, 0.4, (hl, wl, 2)).astype(np.float32)
    T0.requires_grad_(True)
    J0.requires_grad_(True)
    ut = cuda(u).requires_grad_(True)
    E = refine.pyramid_energy(T0, J0, ut, level, ALPHA)
    E.backward()
    Eo = oracle.energy(pyrT[level], pyrJ[level], u, ALPHA)
    guo, gto, gjo = oracle.energy_grad(pyrT[level], pyrJ[level], u, ALPHA)
    shapes = [x.shape for x in pyrT]
    for l in range(level, 0, -1):
        gto = oracle.pyr_down_adjoint(gto, *shapes[l - 1])
        gjo = oracle.pyr_down_adjoint(gjo, *shapes[l - 1])
    assert float(E.detach()) == pytest.approx(Eo, rel=1e-5)
    for got, ref in ((ut.grad, guo), (T0.grad, gto), (J0.grad, gjo)):
        got = got.cpu().numpy()
        assert np.abs(got - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())


def test_refinement_lowers_energy_and_recovers_flow():
    p = synth.pair_small_gray(seed=9, h=256, w=256, amp_x=3.0, amp_y=1.5, levels=3)
    u, trace = refine.refine_flow(cuda(p.L), cuda(p.R), levels=3, steps=40, lr=0.05, alpha=ALPHA)
    torch.cuda.synchronize()
    for level, first, last in trace:
        assert last < first, (level, first, last)
    m = 12
    err = np.hypot(*(u.cpu().numpy() - p.flow_LtoR).transpose(2, 0, 1))[m:-m, m:-m]
    zero = np.hypot(*p.flow_LtoR.transpose(2, 0, 1))[m:-m, m:-m]
    assert err.mean() < 0.35 * zero.mean(), (err.mean(), zero.mean())


def _step_arrays(h, w, level, seed):
    g = np.random.default_rng(seed)
    T = g.uniform(0, 1, (h, w)).astype(np.float32)
    J = (0.7 * T + 0.3 * g.uniform(0, 1, (h, w))).astype(np.float32)
    for _ in range(level):
        h, w = (h + 1) // 2, (w + 1) // 2
    # a smooth flow (neighbouring pixels share taps), some noise, some far out
    u = np.stack(np.broadcast_arrays(1.3 + 0.01 * np.arange(w)[None, :], -0.6 + 0.02 * np.arange(h)[:, None]), -1)
    u = u + g.normal(0, 0.2, u.shape)
    u[:: 7, :: 5] *= 40
    return cuda(T), cuda(J), cuda(u)


@pytest.mark.parametrize("h,w,level", [(1, 1, 0), (1, 40, 0), (33, 31, 0), (64, 65, 0), (9, 257, 1), (37, 53, 1), (2, 3, 1),
                                       (66, 130, 2), (35, 5, 2), (131, 67, 3), (130, 260, 5)])
def test_one_call_steps_equal_the_composed_ones(h, w, level):
    # pano_refine_energy / pano_refine_grad against the same step composed from
    # pano_stage_pyr_down, pano_energy_grad and pano_stage_pyr_down_adjoint;
    # sums and the dE/dJ scatter differ in their order only
    T0, J0, u = _step_arrays(h, w, level, 100 + h)
    T, J = refine._levels(T0, level), refine._levels(J0, level)
    E, gu, gt, gj = binding.energy_grad(T[-1].contiguous(), J[-1].contiguous(), u, ALPHA)
    shapes = [tuple(x.shape) for x in T]
    gt, gj = refine._reduce_transpose(gt, shapes), refine._reduce_transpose(gj, shapes)
    scale = torch.tensor(-2.5, dtype=torch.float64, device=DEV)
    E1 = binding.refine_energy(T0, J0, u, level, ALPHA)
    du, dT, dJ = binding.refine_grad(T0, J0, u, level, ALPHA, scale)
    assert float(E1) == pytest.approx(float(E), rel=1e-12)
    for got, ref in ((du, gu), (dT, gt), (dJ, gj)):
        assert (got - ref * -2.5).abs().max() <= 4e-6 * max(1.0, float(ref.abs().max()))
    only = binding.refine_grad(T0, J0, u, level, ALPHA, None, want_u=False, want_T=False)
    assert only[0] is None and only[1] is None
    assert (only[2] - gj).abs().max() <= 4e-6 * max(1.0, float(gj.abs().max()))


@pytest.mark.parametrize("shape", [(1, 1), (1, 2), (2, 1), (3, 3), (4, 5), (5, 4), (6, 6), (64, 16), (65, 17), (130, 131)])
def test_adjoint_at_the_border_of_its_interior(shape):
    h, w = shape
    g = np.random.default_rng(h * 1000 + w).normal(0, 1, ((h + 1) // 2, (w + 1) // 2)).astype(np.float32)
    got = binding.stage_pyr_down_adjoint(cuda(g), h, w).cpu().numpy()
    # sixteen products of weights that are powers of two times 6 or 11 sixteenths
    np.testing.assert_allclose(got, oracle.pyr_down_adjoint(g, h, w), rtol=0, atol=2e-6)


@pytest.mark.parametrize("factor", [1.0, 1e-12, 1e-18, 1e17, 0.0])
def test_energy_of_very_small_and_large_differences(factor):
    # beyond 1e-12 .. 1e15 the squares are summed in doubles
    g = np.random.default_rng(5)
    T = cuda(np.zeros((70, 90)))
    J = cuda(g.normal(0, 1, (70, 90)) * factor)
    u = cuda(np.zeros((70, 90, 2)))
    E = float(binding.energy_grad(T, J, u, ALPHA, want_u=False, want_T=False, want_J=False)[0])
    assert E == pytest.approx(float((J.double() ** 2).sum()), rel=1e-12)


# More than one tile per thread of the energy's fixed grid (above 311296 pixels),
# up to several rounds of the float sums. The residual does not depend on the
# flow (a constant target), so a float64 sum of the same float32 residuals and
# differences is E up to the order of the double additions: at most 1216 of them
# across CTAs, 31 within one and n / 16 + 1 in a thread, 2^-53 of the sum each.
@pytest.mark.parametrize("factor", [1.0, 1e-16, 1e18])
@pytest.mark.parametrize("kind", ["constant", "random"])
@pytest.mark.parametrize("h,w", [(1031, 777), (2003, 1999), (6007, 4001)])
def test_energy_of_many_pixels_per_thread(h, w, kind, factor):
    if kind == "constant":
        T = torch.full((h, w), 0.3, device=DEV)
        odd = (torch.arange(h, device=DEV)[:, None] + torch.arange(w, device=DEV)) % 2
        u = torch.stack([0.37 * odd, -0.11 * odd], -1).float()
    else:
        g = torch.Generator(device=DEV).manual_seed(h)
        T = torch.rand((h, w), generator=g, device=DEV)
        u = torch.randn((h, w, 2), generator=g, device=DEV)
    T, J, u = T * factor, torch.full((h, w), 0.21 * factor, device=DEV), (u * factor).contiguous()
    E = float(binding.energy_grad(T, J, u, ALPHA, want_u=False, want_T=False, want_J=False)[0])
    sq = lambda d: float((d.double() ** 2).sum())
    ref = sq(J - T) + float(np.float32(ALPHA)) * (sq(u[:, 1:] - u[:, :-1]) + sq(u[1:] - u[:-1]))
    n = h * w / (1216 * 256)
    assert E == pytest.approx(ref, rel=(1216 + 31 + n / 16 + 1) * 2.0 ** -53)


def test_energy_of_non_numbers():
    T, u = cuda(np.zeros((40, 40))), cuda(np.zeros((40, 40, 2)))
    for value, check in ((np.inf, np.isinf), (np.nan, np.isnan)):
        A = np.zeros((40, 40))
        A[39, 39] = value
        # at the corner: every tap of the pixel is the value itself for T; J mixes inf - inf
        E = float(binding.energy_grad(cuda(A), T, u, ALPHA, want_u=False, want_T=False, want_J=False)[0])
        assert check(E)


def _reuse_at_once(sizes):
    """Allocate the sizes (bytes) on the current stream and overwrite them."""
    kept = [torch.full((n,), 0x7F, dtype=torch.uint8, device=DEV) for n in sizes for _ in range(4)]
    torch.cuda.current_stream().synchronize()
    return kept


def test_scratch_of_a_call_on_another_stream():
    # the side stream is busy when the calls return: what the current stream
    # allocates meanwhile must not be their scratch or copies
    h, w, level = 301, 402, 2
    T0, J0, u = _step_arrays(h, w, level, 11)
    u = u.transpose(0, 1).contiguous().transpose(0, 1)      # copied by the call
    E = binding.refine_energy(T0, J0, u, level, ALPHA)
    want = binding.refine_grad(T0, J0, u, level, ALPHA)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    n = int(binding.load_library().pano_refine_scratch_bytes(h, w, level))
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)                       # some 10 ms
    E1 = binding.refine_energy(T0, J0, u, level, ALPHA, stream=side)
    got = binding.refine_grad(T0, J0, u, level, ALPHA, stream=side)
    kept = _reuse_at_once([n, u.numel() * 4])
    side.synchronize()
    assert float(E1) == pytest.approx(float(E), rel=1e-12)
    for a, b in zip(got, want):
        assert (a - b).abs().max() <= 4e-6 * max(1.0, float(b.abs().max()))
    del kept
