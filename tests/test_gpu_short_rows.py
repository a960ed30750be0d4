"""FP64 x pass at the edges of its form for few short rows (at most 64 points, at most
152 rows): lengths around a warp and the limit, all orders, any number of threads,
against torch; planes with a non-finite entry."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1711_01365_gb300 import build
    build.build()
    from paper_1711_01365_gb300 import mbo
    return mbo


def heat(A, dims, tau):
    e = 0.0
    for ax, N in enumerate(dims):
        k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        e = e - 4 * torch.pi ** 2 * tau * (k * k).reshape([-1 if ax == b else 1 for b in range(len(dims))])
    d = tuple(range(1, len(dims) + 1))
    return torch.fft.ifftn(torch.fft.fftn(A, dim=d) * torch.exp(e), dim=d).real


@pytest.mark.parametrize("n", [1, 2, 3, 4])
@pytest.mark.parametrize("dims,threads", [((2, 2), 0), ((3, 32), 0), ((32, 36), 0), ((144, 64), 0), ((144, 72), 0),
                                          ((162, 54), 0), ((9, 16, 27), 0), ((18, 9, 48), 0), ((48, 54), 32),
                                          ((48, 54), 96), ((48, 64), 384), ((16, 16), 352)])
def test_short_rows_match_torch(M, dims, threads, n):
    tau = 3.0 / max(dims) ** 2
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn((n * n,) + dims, generator=g, device="cuda", dtype=torch.float64)
    want = heat(A, dims, tau)
    out, B, P = torch.empty_like(A), A.clone(), torch.empty_like(A)
    h = M.Mbo(dims, n, tau, "f64", row_threads=threads)
    h.diffuse(A, out)
    # both transforms round: a few eps of the field's size times the root of the stages
    assert float((out - want).abs().max()) <= 2e-15 * float(A.abs().max())
    h.step(B)
    h.project(out, P)
    h.close()
    # the fused pass projects the same diffused values; near-singular points magnify rounding
    assert float((B - P).abs().median()) <= 1e-15
    C = B.reshape(n, n, -1).permute(2, 0, 1)
    eye = torch.eye(n, device="cuda", dtype=torch.float64)
    assert float((C.transpose(1, 2) @ C - eye).abs().max()) <= 1e-14


@pytest.mark.parametrize("dims", [(16, 24), (64, 64), (96, 128)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_non_finite_entry_spoils_its_plane_only(M, dims, bad):
    g = torch.Generator(device="cuda").manual_seed(8)
    A = torch.randn((9,) + dims, generator=g, device="cuda", dtype=torch.float64)
    h = M.Mbo(dims, 3, 3.0 / max(dims) ** 2, "f64")
    want, out = torch.empty_like(A), torch.empty_like(A)
    h.diffuse(A, want)
    A[4, 1, 5] = bad  # channels 4 and 5 are one complex plane
    h.diffuse(A, out)
    h.close()
    assert torch.isnan(out[4:6]).all()
    for c in (0, 1, 2, 3, 6, 7, 8):
        assert torch.equal(out[c], want[c])
