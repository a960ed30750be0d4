"""FP64 projection (n = 3) of prescribed matrices, in the fused step and in mbo_project,
against the polar factor in extended precision: random, nearly orthogonal and
graded matrices, both classes, matrices on both sides of the smallest |det| that
the FP32-guided iteration takes, and scales beyond the FP32 range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 32
# RMS of |error|_F: a quarter above what scaled Newton steps leave by rounding alone
# (1.48e-16, 1.29e-16 and 2.0e-16; emulated on the CPU over 60000 matrices each)
RMS = {"random": 1.85e-16, "near": 1.6e-16, "graded": 2.6e-16, "det_edge": None, "det_small": None}


@pytest.fixture(scope="module")
def M():
    from paper_1711_01365_gb300 import build
    build.build()
    from paper_1711_01365_gb300 import mbo
    return mbo


def matrices(kind, g):
    if kind == "random":
        return g.standard_normal((N * N, 3, 3))
    u, v = (np.linalg.qr(g.standard_normal((N * N, 3, 3)))[0] for _ in range(2))
    r = g.uniform(size=(3, N * N))
    if kind == "near":
        s = 1 - 1e-3 * r
    elif kind == "graded":
        s1 = 0.03 + 0.05 * r[0]
        s = np.stack([np.ones(N * N), s1, s1 * (0.05 + 0.95 * r[1])])
    else:  # |det| / |m|_F^3 from 2e-5 to 5e-4, and from 2e-6 to 5e-5: the guided form takes 1e-5 and above
        s1 = 0.05 + 0.9 * r[0]
        nf = np.sqrt(1 + s1 * s1)
        s = np.stack([np.ones(N * N), s1, (2e-5 if kind == "det_edge" else 2e-6) * 25.0 ** r[1] * nf ** 3 / s1])
    return np.einsum("pij,jp,pkj->pik", u, s, v)


def polar(m):
    """Scaled Newton iteration in extended precision."""
    X = m.astype(np.longdouble)
    X /= np.sqrt((X * X).sum((1, 2)))[:, None, None]
    for it in range(40):
        C = np.stack([np.cross(X[:, (i + 1) % 3], X[:, (i + 2) % 3]) for i in range(3)], 1)
        d = (X[:, 0] * C[:, 0]).sum(1)[:, None, None]
        z = (((C / d) ** 2).sum((1, 2)) / (X ** 2).sum((1, 2))) ** np.longdouble(0.25) if it < 28 else np.ones(len(X))
        z = z[:, None, None]
        X = (z * X + C / (z * d)) / 2
    return X


@pytest.mark.parametrize("kind", ["random", "near", "graded", "det_edge", "det_small"])
@pytest.mark.parametrize("scale", [1.0, 1e-13, 1e13])
@pytest.mark.parametrize("fused", [True, False])
def test_projection_error(M, kind, scale, fused):
    m = matrices(kind, np.random.default_rng(11)) * scale
    A = torch.from_numpy(np.ascontiguousarray(m.reshape(-1, 9).T).reshape(9, N, N)).cuda()
    h = M.Mbo((N, N), 3, 1e-14, "f64")  # the heat factor is 1 - 2e-10 at most
    mt, B = torch.empty_like(A), A.clone()
    h.diffuse(A, mt)
    if fused:
        h.step(B)
    else:
        h.project(mt, B)
    h.close()
    mt = mt.cpu().numpy().reshape(9, -1).T.reshape(-1, 3, 3)
    b = B.cpu().numpy().reshape(9, -1).T.reshape(-1, 3, 3).astype(np.longdouble)
    err = np.sqrt(((b - polar(mt)) ** 2).sum((1, 2))).astype(float)
    defect = np.abs(np.einsum("pji,pjk->pik", b, b) - np.eye(3)).max((1, 2)).astype(float)
    s = np.linalg.svd(mt, compute_uv=False)
    cond = np.minimum(1.0, (s[:, 1] + s[:, 2]) / s[:, 0])
    # rounding of m's entries alone moves the factor by eps |m| / (s2 + s3)
    assert (err * cond).max() <= 8e-16
    assert defect.max() <= 8e-16 and defect.mean() <= 1.6e-16
    if RMS[kind]:
        assert np.sqrt((err ** 2).mean()) <= RMS[kind]


@pytest.mark.parametrize("dims", [(48, 64), (72, 72, 96), (512, 96)])
def test_step_statistics_equal_the_unfused_ones(M, dims):
    """n = 3: the fused step's field and records against diffusion, projection and torch."""
    tau = 3.0 / max(dims) ** 2
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randn((9,) + dims, generator=g, device="cuda", dtype=torch.float64)
    h = M.Mbo(dims, 3, tau, "f64")
    h.project(A, A)
    old, At, B = A.clone(), torch.empty_like(A), torch.empty_like(A)
    h.diffuse(old, At)
    h.project(At, B)
    E = h.lyapunov(old)
    rec = h.step(A, want_stats=True)
    h.close()
    det = lambda F: torch.linalg.det(F.reshape(3, 3, -1).permute(2, 0, 1))  # noqa: E731
    assert rec["max_delta"] == float((A - old).abs().max())
    assert rec["det_flips"] == int(((det(A) >= 0) != (det(old) >= 0)).sum())
    assert rec["nonfinite"] == 0
    assert rec["energy"] == pytest.approx(E, rel=1e-12)
    s = torch.linalg.svdvals(At.reshape(3, 3, -1).permute(2, 0, 1))
    clear = (s[:, 2] > 1e-6 * s[:, 0]) & (s[:, 1] + s[:, 2] > 1e-2)
    assert float((A - B).abs().amax(0).reshape(-1)[clear].max()) <= 1e-12
