"""Passes that walk their work with a stride of the grid, and the selection of
the volume-preserving step, at the sizes where such loops can go wrong.

* A projecting x pass over more rows than blocks fit on the GPU (72^2 x 96, and
  4096 two-row groups of 256 points): the step's statistics against the fields
  it read and wrote, its field against the unfused calls.
* The radix selection for n = 1, where dE = 2 A~ and the chosen set is known
  exactly from the diffused field: ties over the whole grid, ties across the
  threshold, every n_plus at the ends of the range and of the 11-bit digits.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1711_01365_gb300 import build
    build.build()
    from paper_1711_01365_gb300 import mbo
    return mbo


@pytest.mark.parametrize("dims,dtype", [((72, 72, 96), "f32"), ((72, 72, 96), "f64"), ((64, 128, 256), "f32"),
                                        ((3, 81), "f64"), ((2, 2), "f32")])
def test_step_statistics_over_many_rows(M, dims, dtype):
    n, tau = 2, 3.0 / max(dims) ** 2
    t = torch.float32 if dtype == "f32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(5)
    raw = torch.randn((n * n,) + dims, generator=g, device="cuda", dtype=torch.float64).to(t)
    h = M.Mbo(dims, n, tau, dtype)
    A = torch.empty_like(raw)
    h.project(raw, A)
    old = A.clone()
    At, B = torch.empty_like(A), torch.empty_like(A)
    h.diffuse(old, At)
    h.project(At, B)
    E = h.lyapunov(old)
    rec = h.step(A, want_stats=True)
    assert rec["max_delta"] == float((A - old).abs().max())
    det = lambda F: F[0] * F[3] - F[1] * F[2]  # noqa: E731
    assert rec["det_flips"] == int(((det(A) >= 0) != (det(old) >= 0)).sum())
    assert rec["energy"] == pytest.approx(E, rel=1e-6 if dtype == "f32" else 1e-12)
    # the fused and the unfused step differ by rounding where the class is clear
    far = (At.double()[0] + At.double()[3]).hypot(At.double()[2] - At.double()[1]) - \
          (At.double()[0] - At.double()[3]).hypot(At.double()[1] + At.double()[2])
    clear = far.abs() > 1e-2
    assert float((A - B).abs().amax(0)[clear].max()) <= (2e-5 if dtype == "f32" else 1e-12)
    h.close()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("dims", [(2, 2), (32, 64), (48, 54), (128, 192)])
@pytest.mark.parametrize("kind", ["constant", "two", "random", "tiny"])
def test_selection_takes_the_largest_lowest_index_first(M, dims, kind, dtype):
    P = int(np.prod(dims))
    r = np.random.default_rng(9)
    F = {"constant": lambda: np.full(dims, 0.25),
         "two": lambda: np.where(np.arange(P).reshape(dims) % dims[1] < dims[1] // 2, 0.5, -0.75),
         "random": lambda: r.standard_normal(dims),
         "tiny": lambda: 1e-30 * r.standard_normal(dims)}[kind]()
    t = torch.float32 if dtype == "f32" else torch.float64
    h = M.Mbo(dims, 1, 4.0 / min(dims) ** 2, dtype)
    A0 = torch.tensor(F, dtype=t, device="cuda")[None].contiguous()
    At = torch.empty_like(A0)
    h.diffuse(A0, At)
    order = np.argsort(-At.cpu().numpy().ravel(), kind="stable")
    for n_plus in sorted({0, 1, P // 3, min(2047, P), min(2048, P), P - 1, P}):
        A = A0.clone()
        h.step_volume(A, n_plus)
        want = -np.ones(P)
        want[order[:n_plus]] = 1.0
        assert np.array_equal(A.cpu().numpy().ravel(), want), n_plus
    A = A0.clone()  # the volume of the field itself
    h.step_volume(A, -1)
    assert int((A > 0).sum()) == int((A0 > 0).sum())
    h.close()


@pytest.mark.parametrize("dims", [(486, 18), (243, 9), (162, 27), (81, 6), (54, 36), (9, 2), (27, 3),
                                  (12, 1458), (1944, 6), (4, 9, 81), (18, 27, 12), (648, 54)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_network_radices_and_ragged_tiles(M, dims, dtype):
    """Axes with every radix of the network's plans, and rows that end in a ragged column tile: the
    diffusion with and without a handle, and the energy, against torch in FP64."""
    n, tau = 2, 3.0 / max(dims) ** 2
    t = torch.float32 if dtype == "f32" else torch.float64
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn((n * n,) + dims, generator=g, device="cuda", dtype=torch.float64).to(t)
    e = 0.0
    for ax, N in enumerate(dims):
        k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        e = e - 4 * np.pi ** 2 * tau * (k * k).reshape([-1 if ax == b else 1 for b in range(len(dims))])
    F = torch.fft.fftn(A.double(), dim=tuple(range(1, len(dims) + 1)))
    want = torch.fft.ifftn(F * torch.exp(e), dim=tuple(range(1, len(dims) + 1))).real
    P = float(np.prod(dims))
    E = float((-torch.expm1(e) * F.abs().square()).sum() / P + (n - A.double().square().sum(0)).sum()) / (P * tau)
    h = M.Mbo(dims, n, tau, dtype)
    out = torch.empty_like(A)
    h.diffuse(A, out)
    tol = 4e-6 if dtype == "f32" else 1e-13
    scale = float(want.abs().max())
    assert float((out.double() - want).abs().max()) <= tol * max(1.0, scale)
    M.mbo_diffuse_noalloc(dims, n, tau, M.MBO_F32 if dtype == "f32" else M.MBO_F64, A, out)
    assert float((out.double() - want).abs().max()) <= tol * max(1.0, scale)
    scaleE = float((F.abs().square().sum() / P + A.double().square().sum())) / (P * tau)
    assert abs(h.lyapunov(A) - E) <= (1e-5 if dtype == "f32" else 1e-12) * scaleE
    h.close()


@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("dims", [(2, 2), (3, 16), (6, 1536), (9, 2048), (2048, 2), (18, 54, 12), (1024, 1024)])
@pytest.mark.parametrize("scale", [1.0, 1e-200, 1e200, 1e-320])
def test_fixed_point_diffusion_is_scale_free(M, dims, n, scale):
    """The FP64 transforms run in fixed point on a scale of their own per sequence: any finite magnitude,
    one channel far below its partner, one bright point, constant fields; and a non-finite value still
    reaches what a floating-point transform would make of it."""
    if scale != 1.0 and np.prod(dims) > 50000:
        pytest.skip("sizes are covered at scale 1")
    if n == 4 and dims[-1] == 2048:
        pytest.skip("rows of eight FP64 planes exceed the shared memory")
    tau = 3.0 / max(dims) ** 2
    g = torch.Generator(device="cuda").manual_seed(11)
    A = torch.randn((n * n,) + dims, generator=g, device="cuda", dtype=torch.float64)
    A[0] += 3.0
    A.view(n * n, -1)[-1, 5 % A[0].numel()] = 1e4
    if n > 1:
        A[1] *= 1e-9
        A[2] = 0.75
    e = 0.0
    for ax, N in enumerate(dims):
        k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        e = e - 4 * np.pi ** 2 * tau * (k * k).reshape([-1 if ax == b else 1 for b in range(len(dims))])
    d = tuple(range(1, len(dims) + 1))
    want = torch.fft.ifftn(torch.fft.fftn(A, dim=d) * torch.exp(e), dim=d).real
    h = M.Mbo(dims, n, tau, "f64")
    out = torch.empty_like(A)
    h.diffuse(A * scale, out)
    if scale == 1e-320:  # denormals keep no digits: nothing but their size is asked
        assert float(out.abs().max()) <= 1e-310
    else:
        rms = want.square().mean(dim=d, keepdim=True).sqrt()
        pair = torch.maximum(rms[0::2], torch.cat([rms[1::2], rms[-1:]])[: rms[0::2].shape[0]])
        lim = 3e-15 * torch.repeat_interleave(pair, 2, dim=0)[: n * n] * np.log2(A[0].numel() + 2)
        assert bool(((out / scale - want).abs() <= lim).all())
    bad = A.clone()
    bad.view(n * n, -1)[0, 3 % A[0].numel()] = float("nan") if n % 2 else float("inf")
    h.diffuse(bad, out)
    assert not bool(torch.isfinite(out[0]).any())
    if n > 2:
        assert bool(torch.isfinite(out[2:]).all())  # the other planes are not touched
    h.close()
