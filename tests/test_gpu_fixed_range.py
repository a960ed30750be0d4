"""FP64 diffusion of fields near the bottom of the FP64 range: subnormal entries,
spectra and results are kept as FP64 arithmetic keeps them (gradual underflow)."""
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


@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("dims", [(2, 2), (48, 54), (6, 1536), (18, 54, 12)])
@pytest.mark.parametrize("e2", [-990, -1000, -1015, -1022, -1030, -1045, -1060])
@pytest.mark.parametrize("noalloc", [False, True])
def test_small_magnitudes_keep_their_digits(M, dims, n, e2, noalloc):
    tau = 3.0 / max(dims) ** 2
    g = torch.Generator(device="cuda").manual_seed(2)
    A = torch.randn((n * n,) + dims, generator=g, device="cuda", dtype=torch.float64).clamp(-6, 6)
    A[0] *= 1e-3  # entries far below their plane's largest one
    ulp = 2.0 ** (-1074 - e2)  # the smallest subnormal, in units of the scale
    tiny = A * 2.0 ** -600 * 2.0 ** (e2 + 600)
    back = lambda t: t * 2.0 ** 600 * 2.0 ** (-e2 - 600)  # noqa: E731
    e = 0.0
    for ax, N in enumerate(dims):
        k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        e = e - 4 * np.pi ** 2 * tau * (k * k).reshape([-1 if ax == b else 1 for b in range(len(dims))])
    d = tuple(range(1, len(dims) + 1))
    want = torch.fft.ifftn(torch.fft.fftn(back(tiny), dim=d) * torch.exp(e), dim=d).real
    out = torch.empty_like(A)
    if noalloc:
        M.mbo_diffuse_noalloc(dims, n, tau, M.MBO_F64, tiny, out)
    else:
        h = M.Mbo(dims, n, tau, "f64")
        h.diffuse(tiny, out)
        h.close()
    # a normal field's error, plus half a smallest subnormal for every rounded value: the spectra
    # that the unnormalised inverse transforms (all axes but the last pass's) sum up, and the result
    rounded = 1 + np.prod(dims[1:])
    lim = 3e-15 * np.log2(A[0].numel() + 2) * float(want.square().mean().sqrt()) + ulp * rounded
    assert float((back(out) - want).abs().max()) <= lim
