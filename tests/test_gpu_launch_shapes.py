"""mbo_launch_config reports the tile width that the network strided passes take, and a
handle created with the reported shapes takes them again; the autotuner does not
leave the automatic shapes for slower ones."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FIELDS = ("row_threads", "axis_threads", "axis_tx", "axis_stages")


@pytest.fixture(scope="module")
def M():
    from paper_1711_01365_gb300 import build
    build.build()
    from paper_1711_01365_gb300 import mbo
    return mbo


def shapes(M, h):
    c = M.mbo_launch_config(h.h)
    return {k: c[k] for k in FIELDS}


def step_us(M, pairs):
    """us per step of each (handle, field), the best of runs taken in turn."""
    e0, e1 = torch.cuda.Event(True), torch.cuda.Event(True)
    best = [float("inf")] * len(pairs)
    for h, A in pairs:
        h.step(A)
    for _ in range(12):
        for i, (h, A) in enumerate(pairs):
            e0.record()
            for _ in range(30):
                h.step(A, M.MBO_STEP_CONTINUE)
            e1.record()
            e1.synchronize()
            best[i] = min(best[i], e0.elapsed_time(e1) / 30 * 1e3)
    return best


# width: what the passes take where that may be given back (it divides nx)
@pytest.mark.parametrize("dims,n,dtype,width", [((128, 128), 2, "f64", 1), ((96, 96), 3, "f32", 2),
                                                ((648, 486), 3, "f32", None), ((512, 243), 3, "f64", None),
                                                ((54, 54, 54), 3, "f32", None), ((1024, 1024), 3, "f64", 4),
                                                ((18, 18), 2, "f64", 1)])
def test_reported_shapes_can_be_given_back(M, dims, n, dtype, width):
    tau = 3.0 / min(dims) ** 2
    A = torch.randn((n * n,) + dims, device="cuda", dtype=torch.float64 if dtype == "f64" else torch.float32)
    h = M.Mbo(dims, n, tau, dtype)
    h.project(A, A)
    s = shapes(M, h)
    if width:
        assert s["axis_tx"] == width
    g = M.Mbo(dims, n, tau, dtype, **s)
    assert shapes(M, g) == s
    B = A.clone()
    t = step_us(M, [(h, A), (g, B)])
    h.close()
    g.close()
    assert t[1] <= 1.06 * t[0] + 1.0, t
    assert torch.equal(A, B)


@pytest.mark.parametrize("dims,n", [((96, 96, 96), 3), ((54, 54, 54), 3), ((81, 81, 81), 3), ((162, 162), 3)])
def test_autotuned_shapes_are_not_slower(M, dims, n):
    tau = 3.0 / min(dims) ** 2
    A = torch.randn((n * n,) + dims, device="cuda")
    h = M.Mbo(dims, n, tau, "f32")
    h.project(A, A)
    g = M.Mbo(dims, n, tau, "f32", autotune=1)
    t = step_us(M, [(h, A), (g, A.clone())])
    h.close()
    g.close()
    assert t[1] <= 1.06 * t[0] + 1.0, t
