"""The FP32 surface diffusion on the points' box of the grid, at the shapes where
the box and the column segments can go wrong: a grid so small that footprints
wrap around it (the box is then whole axes), points on one line or in one spot,
a single point, more sources in one footprint start than a segment holds, and
every order n and kernel width, against the oracle's double sum."""
import numpy as np
import pytest

from oracle import surface as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    from paper_1711_01365_gb300 import build
    build.build()
    from paper_1711_01365_gb300 import mbo
    return mbo


def points(kind, nq):
    g = np.random.default_rng(4)
    if kind == "cube":
        x = g.uniform(0, 1, (nq, 3))
    elif kind == "line":
        x = np.stack([g.uniform(0, 1, nq), np.full(nq, 0.3), np.full(nq, -2.0)], 1)
    elif kind == "spot":  # all but a few sources share a footprint start
        x = 0.5 + 1e-4 * g.standard_normal((nq, 3))
        x[:3] = g.uniform(0, 1, (3, 3))
    else:
        x = np.array([[0.2, -0.1, 3.0]])
    c = x + (0.01 * g.standard_normal(x.shape) if kind != "point" else 0.0)
    return x, g.uniform(0.5, 1.5, len(x)) / len(x), c


@pytest.mark.parametrize("n,eps", [(1, 1e-6), (2, 1e-6), (3, 1e-6), (4, 1e-6), (3, 1e-4), (2, 1e-7)])
@pytest.mark.parametrize("kind,tau", [("cube", 0.5), ("cube", 0.01), ("line", 0.01), ("spot", 0.02), ("point", 0.05)])
def test_box_diffusion_matches_the_double_sum(M, kind, tau, n, eps):
    xq, wq, xc = points(kind, 700)
    A = np.random.default_rng(8).standard_normal((n * n, len(wq)))
    s = M.Surface(xq, wq, xc, n, tau, eps, "f32")
    p = s.params()
    want = S.surface_diffuse(A, xq, wq, xc, tau, p["h"], p["M"])
    a = torch.tensor(A, dtype=torch.float32, device="cuda")
    out = s.diffuse(a, torch.empty_like(a)).double().cpu().numpy()
    # the spreading error is eps of the sum of the magnitudes, about 0.8 (4 pi tau)^(-3/2) for unit weights
    scale = max(np.abs(want).max(), 0.2 * (4 * np.pi * tau) ** -1.5)
    assert np.abs(out - want).max() <= max(2e-5, 20 * eps) * scale
    s.close()
