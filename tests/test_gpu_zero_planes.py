"""FP64 fields with zero channels take no longer than full ones (a sequence of zeros
needs no scale), and their results stay exact zeros."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1711_01365_gb300 import build
    build.build()
    from paper_1711_01365_gb300 import mbo
    return mbo


def per_call(calls, k=20):
    """ms per call of each, the best of runs taken in turn."""
    e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
    best = [float("inf")] * len(calls)
    for _ in range(10):
        for i, f in enumerate(calls):
            e0.record()
            for _ in range(k):
                f()
            e1.record()
            e1.synchronize()
            best[i] = min(best[i], e0.elapsed_time(e1) / k)
    return best


@pytest.mark.parametrize("dims,n", [((96, 96, 96), 3), ((96, 96, 54), 3)])
def test_zero_channels_cost_no_more(M, dims, n):
    full = torch.randn((n * n,) + dims, device="cuda", dtype=torch.float64)
    phases = torch.zeros_like(full)
    for i in range(n):
        phases[i * n + i] = 1.0
    phases[0, ..., : dims[-1] // 2] = -1.0
    out = torch.empty_like(full)
    h = M.Mbo(dims, n, 3.0 / min(dims) ** 2, "f64")
    t = per_call([lambda: h.diffuse(full, out), lambda: h.diffuse(phases, out)])
    # channels 2q and 2q + 1 share a plane: both zero
    zero = [c for c in range(n * n - 1) if c % 2 == 0 and not phases[c:c + 2].any()]
    for c in zero:
        assert not out[c:c + 2].any()
    h.close()
    assert t[1] <= 1.1 * t[0], t


@pytest.mark.parametrize("dims", [(6, 6), (48, 54), (18, 54, 12)])
@pytest.mark.parametrize("scale", [1.0, 1e-40, 1e200])
def test_zero_columns_beside_live_ones(M, dims, scale):
    """One live line in a field of zeros: its tile holds zero columns and a scaled one."""
    n, tau = 2, 3.0 / max(dims) ** 2
    A = torch.zeros((4,) + dims, device="cuda", dtype=torch.float64)
    A[0].reshape(-1, dims[-1])[:, 1] = torch.randn(A[0].numel() // dims[-1], device="cuda", dtype=torch.float64)
    A[3] = A[0] * 1e-3
    want = torch.zeros_like(A)
    e = 0.0
    for ax, N in enumerate(dims):
        k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        e = e - 4 * torch.pi ** 2 * tau * (k * k).reshape([-1 if ax == b else 1 for b in range(len(dims))])
    for c in range(4):
        want[c] = torch.fft.ifftn(torch.fft.fftn(A[c]) * torch.exp(e)).real
    out = torch.empty_like(A)
    h = M.Mbo(dims, n, tau, "f64")
    h.diffuse(A * scale, out)
    h.close()
    lim = 3e-15 * float(want.abs().max())
    assert float((out / scale - want).abs().max()) <= lim


@pytest.mark.parametrize("dims,n", [((16, 16), 3), ((96, 128), 3), ((96, 128), 2)])
def test_step_of_subnormal_phases(M, dims, n):
    """The projection does not depend on the scale: two constant phases times 2^-1030,
    most channels zero, step like the phases themselves."""
    A = torch.zeros((n * n,) + dims, device="cuda", dtype=torch.float64)
    for i in range(n):
        A[i * n + i] = 1.0
    A[0, ..., : dims[-1] // 2] = -1.0
    B = A * 2.0 ** -600 * 2.0 ** -430
    h = M.Mbo(dims, n, 3.0 / min(dims) ** 2, "f64")
    h.step(A)
    h.step(B)
    h.close()
    assert float((A - B).abs().max()) <= 1e-9
