"""The work that is timed: steps, runs, batches, volume steps and surface steps.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (the fields, on the GPU, and the handle), ``run`` makes the
call, ``exact`` gives the same outputs from plain 64-bit torch, and ``work``
counts what a pass cannot do without.  Sizes are those of the repository's
workloads (128^2, 1024^2, 256^3, 512^3, the mixed batch, the unit sphere) and
others of the same kinds.  Fields are O(n)-valued, as Algorithm 1 has them:

``gauss``    iid N(0, 1) matrices, det > 0 on x < 1/2 and det < 0 elsewhere,
             projected onto O(n) by the library, as the FP64 workloads start.
``regions``  a smooth rotation field, reflected inside a smooth random region:
             two phases with an interface, what an evolution looks like after
             its first steps.
``specks``   a smooth rotation field with a tenth of the points replaced by
             random matrices of determinant -1 (the 3-D workloads' initial field).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1711_01365_gb300 import mbo

# Axis lengths (2^a 3^b) that the drawn cases take.
LENGTHS = (48, 54, 64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256, 288, 324, 384, 432, 486,
           512, 576, 648, 729, 768, 864, 972, 1024, 1152, 1296, 1458, 1536, 1728, 1944, 2048)
BATCH_SIZES = (256, 384, 512, 768, 1024, 1536, 2048)


def listed():
    return [
        # the smallest workload: a whole FP64 run of a small O(2) field (graph replay, launches count)
        {"name": "run_128_n2_f64", "kind": "run", "dims": "128,128", "n": 2, "dtype": "f64", "field": "gauss",
         "tau": 4.0, "steps": 16},
        # one steady-state step of a small field: latency
        {"name": "step_256_n2_f32", "kind": "step", "dims": "256,256", "n": 2, "dtype": "f32",
         "field": "regions", "tau": 4.0},
        # a run of an ordinary field with its energies and flip counts read back
        {"name": "run_512_n3_f32", "kind": "run", "dims": "512,512", "n": 3, "dtype": "f32",
         "field": "regions", "tau": 4.0, "steps": 24},
        # the headline workload's step, and its FP64 form
        {"name": "step_1024_n3_f32", "kind": "step", "dims": "1024,1024", "n": 3, "dtype": "f32",
         "field": "regions", "tau": 3.0},
        {"name": "step_1024_n3_f64", "kind": "step", "dims": "1024,1024", "n": 3, "dtype": "f64",
         "field": "gauss", "tau": 3.0},
        # ragged sizes: radix-3 axes that are not powers of two times three
        {"name": "step_486x648_n3_f32", "kind": "step", "dims": "486,648", "n": 3, "dtype": "f32",
         "field": "regions", "tau": 3.0},
        # a 2-D field larger than L2
        {"name": "step_1536x2048_n3_f32", "kind": "step", "dims": "1536,2048", "n": 3, "dtype": "f32",
         "field": "regions", "tau": 3.0},
        # the 3-D workloads
        {"name": "step_256cubed_n3_f32", "kind": "step", "dims": "256,256,256", "n": 3, "dtype": "f32",
         "field": "specks", "tau": 2.0},
        {"name": "step_512cubed_n3_f32", "kind": "step", "dims": "512,512,512", "n": 3, "dtype": "f32",
         "field": "specks", "tau": 2.0},
        # many independent fields of uneven sizes and orders in one call
        {"name": "batch_28_f32", "kind": "batch", "count": 28, "first": 0, "dtype": "f32", "field": "specks",
         "tau": 4.0},
        # the volume-preserving step of the paper's flat-torus experiment (1024^2, n = 2)
        {"name": "volume_1024_n2_f32", "kind": "volume", "dims": "1024,1024", "n": 2, "dtype": "f32",
         "field": "regions", "tau": 8.0},
        # the closed-surface step: unit sphere, the paper's spacing and tau, 3.3 million points
        {"name": "sphere_005_n3_f32", "kind": "sphere", "dx": 0.05, "p": 3, "n": 3, "dtype": "f32"},
    ]


def draw(rng):
    kind = rng.choice(("step2", "step2", "step2", "step3", "run", "batch", "volume", "sphere"))
    def axis(lo, hi):
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min(LENGTHS, key=lambda v: abs(math.log(v / want)))
    n = rng.choice((2, 3))
    if kind == "step2":
        f64 = rng.random() < 0.3
        dims = [axis(128, 1024 if f64 else 2048) for _ in range(2)]
        return {"kind": "step", "dims": "%d,%d" % tuple(dims), "n": n, "dtype": "f64" if f64 else "f32",
                "field": "gauss" if f64 else "regions", "tau": rng.choice((2.0, 3.0, 4.0))}
    if kind == "step3":
        dims = [axis(48, 384) for _ in range(3)]
        return {"kind": "step", "dims": "%d,%d,%d" % tuple(dims), "n": n, "dtype": "f32", "field": "specks",
                "tau": rng.choice((2.0, 3.0))}
    if kind == "run":
        f64 = rng.random() < 0.5
        dims = [axis(64, 256 if f64 else 768) for _ in range(2)]
        return {"kind": "run", "dims": "%d,%d" % tuple(dims), "n": n, "dtype": "f64" if f64 else "f32",
                "field": "gauss" if f64 else "regions", "tau": rng.choice((3.0, 4.0)),
                "steps": rng.randint(8, 24)}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(8, 28), "first": rng.randint(0, 6), "dtype": "f32",
                "field": "specks", "tau": rng.choice((2.0, 3.0, 4.0))}
    if kind == "volume":
        dims = [axis(128, 1024) for _ in range(2)]
        return {"kind": "volume", "dims": "%d,%d" % tuple(dims), "n": n, "dtype": "f32", "field": "regions",
                "tau": rng.choice((4.0, 8.0))}
    return {"kind": "sphere", "dx": round(rng.uniform(0.07, 0.15), 4), "p": rng.choice((2, 3)), "n": n,
            "dtype": "f32"}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _dims(case):
    return tuple(int(v) for v in case["dims"].split(","))


def _tau(case, dims):
    """The diffusion time: so many squares of the coarsest grid spacing."""
    return case["tau"] / min(dims) ** 2


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _smooth(coords, amp, g, kmax, modes=6):
    """A sum of random plane waves at the given coordinates (broadcast), std `amp`."""
    k = torch.randint(-kmax, kmax + 1, (modes, len(coords)), generator=g, device="cuda").tolist()
    ph = (2 * math.pi * torch.rand(modes, generator=g, device="cuda")).tolist()
    out = 0.0
    for m in range(modes):
        if not any(k[m]):
            k[m][0] = 1
        arg = ph[m]
        for c, x in enumerate(coords):
            arg = arg + (2 * math.pi * k[m][c]) * x
        out = out + torch.cos(arg)
    return out * (amp * math.sqrt(2.0 / modes))


def _rotations(n, comps):
    """exp of the antisymmetric matrices with these components: a list of n*n tensors."""
    if n == 2:
        c, s = torch.cos(comps[0]), torch.sin(comps[0])
        return [c, -s, s, c.clone()]
    wx, wy, wz = comps
    t = torch.sqrt(wx * wx + wy * wy + wz * wz).clamp_min(1e-12)
    x, y, z = wx / t, wy / t, wz / t
    s, c = torch.sin(t), 1 - torch.cos(t)
    return [1 - c * (y * y + z * z), c * x * y - s * z, c * x * z + s * y,
            c * x * y + s * z, 1 - c * (x * x + z * z), c * y * z - s * x,
            c * x * z - s * y, c * y * z + s * x, 1 - c * (x * x + y * y)]


def _speck(F, n, g):
    """Replace a tenth of the points by random matrices of determinant -1."""
    flat = F.view(n * n, -1)
    idx = (torch.rand(flat.shape[1], generator=g, device="cuda") < 0.1).nonzero().squeeze(1)
    if n == 2:
        a = 2 * math.pi * torch.rand(idx.numel(), generator=g, device="cuda")
        flat[:, idx] = torch.stack([torch.cos(a), torch.sin(a), torch.sin(a), -torch.cos(a)]).to(F.dtype)
    else:
        w, x, y, z = torch.nn.functional.normalize(
            torch.randn(4, idx.numel(), generator=g, device="cuda"), dim=0)
        R = [1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
             2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
             2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]
        flat[:, idx] = -torch.stack(R).to(F.dtype)


def _field(kind, dims, n, dtype, seed):
    """The raw field of a torus case (gauss: not yet projected), shape (n*n, *dims)."""
    g = _gen(seed)
    if kind == "gauss":
        F = torch.randn((n, n) + dims, generator=g, device="cuda", dtype=torch.float64)
        want = torch.where(torch.arange(dims[-1], device="cuda") < dims[-1] // 2, 1.0, -1.0).double()
        wrong = _det(F.reshape((n * n,) + dims), n) * want < 0
        F[:2] = torch.where(wrong, F[[1, 0]], F[:2])
        return F.reshape((n * n,) + dims).to(dtype).contiguous()
    coords = [(torch.arange(N, device="cuda", dtype=torch.float32) / N).reshape(
        [-1 if a == b else 1 for b in range(len(dims))]) for a, N in enumerate(dims)]
    comps = [_smooth(coords, 0.8, g, 3).expand(dims) for _ in range(1 if n == 2 else 3)]
    ch = _rotations(n, comps)
    del comps
    F = torch.empty((n * n,) + dims, dtype=dtype, device="cuda")
    for i, c in enumerate(ch):
        F[i] = c
    del ch
    if kind == "regions":
        inside = _smooth(coords, 1.0, g, 2) > 0.3
        for i in range(n):
            F[i * n + n - 1] = torch.where(inside, -F[i * n + n - 1], F[i * n + n - 1])
    else:
        _speck(F, n, g)
    return F


@functools.lru_cache(maxsize=2)
def _band(dx, p):
    """Quadrature points, weights and closest points of the unit sphere's band."""
    tau = 2.0 * dx * dx  # the paper's ratio: dx = 0.05, tau = 0.005
    wb = mbo.mbo_surface_band_width(1e-6, tau)
    return mbo.mbo_surface_sphere_band(1.0, dx, wb, p) + (tau,)


def _surface_field(case, xc, seed):
    n = int(case["n"])
    g = _gen(seed)
    x = torch.from_numpy(np.ascontiguousarray(xc.T)).cuda().float()
    coords = [x[a] * 0.25 for a in range(3)]
    comps = [_smooth(coords, 0.8, g, 3) for _ in range(1 if n == 2 else 3)]
    F = torch.stack(_rotations(n, comps)).contiguous()
    _speck(F, n, g)
    return F


def _batch_list(case):
    out = []
    for i in range(case["count"]):
        N = BATCH_SIZES[(i + case["first"]) % len(BATCH_SIZES)]
        out.append(((N, N), 2 + i % 2, case["tau"] / N ** 2))
    return out


# --------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        fl = _batch_list(case)
        fields = [_field(case["field"], d, n, torch.float32, seed * 64 + i) for i, (d, n, _) in enumerate(fl)]
        return {"case": case, "A": fields, "on": False,
                "h": mbo.Batch([d for d, _, _ in fl], [n for _, n, _ in fl], [t for _, _, t in fl], dtype="f32")}
    if kind == "sphere":
        xq, wq, xc, tau = _band(case["dx"], case["p"])
        return {"case": case, "A": _surface_field(case, xc, seed),
                "h": mbo.Surface(xq, wq, xc, case["n"], tau, 1e-6, dtype=case["dtype"])}
    dims = _dims(case)
    h = mbo.Mbo(dims, case["n"], _tau(case, dims), dtype=case["dtype"])
    A = _field(case["field"], dims, case["n"], _dtype(case), seed)
    if case["field"] == "gauss":
        h.project(A, A)
    return {"case": case, "A": A, "h": h, "on": False}


def run(state):
    case, h, A = state["case"], state["h"], state["A"]
    kind = case["kind"]
    if kind in ("step", "batch"):  # a loop of steps: all but the first continue
        h.step(A, mbo.MBO_STEP_CONTINUE if state["on"] else 0)
        state["on"] = True
        return A
    if kind == "run":  # never stops early, so that every pass does the same number of steps
        r = h.run(A, case["steps"], -1.0)
        f = np.float64 if case["dtype"] == "f64" else np.float32  # the records carry the field's precision
        return {"A": A, "energies": r["energies"].astype(f), "max_deltas": r["max_deltas"].astype(f),
                "det_flips": r["det_flips"]}
    if kind == "volume":  # keeps the number of points of positive determinant
        h.step_volume(A, -1)
        return A
    h.step(A)
    return A


def work(case):
    """Each step reads its field and writes the new one; the transforms, the polar factor and the
    statistics are counted as flops (5 log2 N a point, plane and transform; 25 n^2 a projection)."""
    kind = case["kind"]
    w = 8 if case["dtype"] == "f64" else 4
    if kind == "sphere":
        xq, wq, xc, _ = _band(case["dx"], case["p"])
        nq, C = wq.size, case["n"] ** 2
        # spreading and interpolation: 7^3 points, two operations, each channel (eps = 1e-6)
        return {"bytes": 2.0 * nq * C * w, "flops": nq * (4.0 * 343 * C + 25 * C)}
    fields = [(d, n) for d, n, _ in _batch_list(case)] if kind == "batch" else [(_dims(case), case["n"])]
    b = f = 0.0
    for d, n in fields:
        P, C = float(np.prod(d)), n * n
        b += 2 * P * C * w
        f += P * (2 * (C / 2) * 5 * math.log2(P) + 25 * C)
    k = case.get("steps", 1)
    return {"bytes": b * k, "flops": f * k}


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _det(m, n):
    if n == 2:
        return m[0] * m[3] - m[1] * m[2]
    return (m[0] * (m[4] * m[8] - m[5] * m[7]) - m[1] * (m[3] * m[8] - m[5] * m[6])
            + m[2] * (m[3] * m[7] - m[4] * m[6]))


def _classes2(m):
    """n = 2: nearest rotation, nearest reflection and the difference of their inner products with m."""
    p, q, r, t = m[0] + m[3], m[2] - m[1], m[0] - m[3], m[1] + m[2]
    rho, sig = torch.hypot(p, q), torch.hypot(r, t)
    rot = torch.stack([p / rho, -q / rho, q / rho, p / rho])
    ref = torch.stack([r / sig, t / sig, t / sig, -r / sig])
    return rot, ref, rho - sig


def _polar(m, n):
    """U V^t of every point (the polar factor): closed form, or scaled Newton iterations."""
    if n == 2:
        rot, ref, d = _classes2(m)
        return torch.where(d >= 0, rot, ref)
    out = torch.empty_like(m)
    flat, of = m.reshape(9, -1), out.view(9, -1)
    step = 1 << 22
    for a in range(0, flat.shape[1], step):
        X = flat[:, a:a + step].clone()
        for it in range(14):
            C = torch.stack([X[4] * X[8] - X[5] * X[7], X[5] * X[6] - X[3] * X[8], X[3] * X[7] - X[4] * X[6],
                             X[2] * X[7] - X[1] * X[8], X[0] * X[8] - X[2] * X[6], X[1] * X[6] - X[0] * X[7],
                             X[1] * X[5] - X[2] * X[4], X[2] * X[3] - X[0] * X[5], X[0] * X[4] - X[1] * X[3]])
            C /= X[0] * C[0] + X[1] * C[1] + X[2] * C[2]
            z = (C.square().sum(0) / X.square().sum(0)) ** 0.25 if it < 9 else 1.0
            X = 0.5 * (z * X + C / z)
        of[:, a:a + step] = X
    return out


def _heat(dims, tau):
    g = torch.zeros((1,) * len(dims), dtype=torch.float64, device="cuda")
    for a, N in enumerate(dims):
        k = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        g = g + (k * k).reshape([-1 if a == b else 1 for b in range(len(dims))])
    return -4 * math.pi ** 2 * tau * g


def _diffuse(A, dims, tau):
    e = torch.exp(_heat(dims, tau))
    out = torch.empty_like(A)
    for c in range(A.shape[0]):
        out[c] = torch.fft.ifftn(torch.fft.fftn(A[c]) * e).real
    return out


def _energy(A, n, dims, tau):
    P = float(np.prod(dims))
    om = -torch.expm1(_heat(dims, tau))
    s = sum(float((om * torch.fft.fftn(A[c]).abs().square()).sum()) for c in range(A.shape[0]))
    return (s / P + float((n - A.square().sum(0)).sum())) / (P * tau)


def _exact_surface(case, seed):
    xq, wq, xc, tau = _band(case["dx"], case["p"])
    n, nq = int(case["n"]), wq.size
    C, eps = n * n, 1e-6
    # spacing and modes of the heat-kernel approximation (Sec. 5.2)
    lo = np.minimum(xq.min(0), xc.min(0))
    hi = np.maximum(xq.max(0), xc.max(0))
    R = float((hi - lo).max())
    h = min(math.pi / R, math.pi / (2 * math.sqrt(tau * abs(math.log(eps)))))
    M = math.ceil(math.sqrt(math.log(2 * h * math.sqrt(tau) / (math.sqrt(math.pi) * eps)) / tau) / h)
    if nq * (2.0 * M) ** 3 * C > 4e11:
        return None  # the plain double sum takes minutes
    A = _surface_field(case, xc, seed).double()
    ctr = 0.5 * (lo + hi)
    m = torch.arange(-M, M, device="cuda", dtype=torch.float64)
    src, dst, w = (torch.from_numpy(v).cuda() for v in (h * (xq - ctr), h * (xc - ctr), wq))
    F = torch.zeros((2 * M, 2 * M, C, 2 * M), dtype=torch.complex128, device="cuda")  # x, y, channel, z
    step = 1 << 15
    for a in range(0, nq, step):
        e = [torch.exp(-1j * src[a:a + step, i, None] * m) for i in range(3)]
        az = ((A[:, a:a + step] * w[a:a + step]).T[:, :, None] * e[2][:, None, :]).reshape(-1, C * 2 * M)
        for i in range(2 * M):
            F[i] += ((e[1] * e[0][:, i:i + 1]).T @ az).view(2 * M, C, 2 * M)
    g = torch.exp(-h * h * tau * m * m)
    F *= (g[:, None, None, None] * g[:, None, None] * g) * (h / (2 * math.pi)) ** 3
    out = torch.empty((C, nq), dtype=torch.float64, device="cuda")
    G = F.reshape(2 * M, -1)
    for a in range(0, nq, step):
        e = [torch.exp(1j * dst[a:a + step, i, None] * m) for i in range(3)]
        b = e[0].shape[0]
        s = torch.zeros((b, C), dtype=torch.complex128, device="cuda")
        for i in range(2 * M):
            v = (e[1] * e[0][:, i:i + 1]) @ F[i].reshape(2 * M, C * 2 * M)
            s += (v.view(b, C, 2 * M) * e[2][:, None, :]).sum(2)
        out[:, a:a + step] = s.real.T
    del G
    return _polar(out, n)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sphere":
        return _exact_surface(case, seed)
    if kind == "batch":
        out = []
        for i, (d, n, tau) in enumerate(_batch_list(case)):
            A = _field(case["field"], d, n, torch.float32, seed * 64 + i).double()
            out.append(_polar(_diffuse(A, d, tau), n))
        return out
    dims, n = _dims(case), case["n"]
    tau = _tau(case, dims)
    A = _field(case["field"], dims, n, _dtype(case), seed).double()
    if case["field"] == "gauss":
        A = _polar(A, n)
    if kind == "step":
        return _polar(_diffuse(A, dims, tau), n)
    if kind == "run":
        en, md, fl = [_energy(A, n, dims, tau)], [], []
        for _ in range(case["steps"]):
            B = _polar(_diffuse(A, dims, tau), n)
            md.append(float((B - A).abs().max()))
            fl.append(int(((_det(B, n) >= 0) != (_det(A, n) >= 0)).sum()))
            A = B
            en.append(_energy(A, n, dims, tau))
        return {"A": A, "energies": np.array(en), "max_deltas": np.array(md),
                "det_flips": np.array(fl, dtype=np.int64)}
    # volume: the n_plus points of largest dE (lower index first) take the closest matrix of SO(n)
    n_plus = int((_det(A, n) > 0).sum())
    m = _diffuse(A, dims, tau).reshape(n * n, -1)
    if n == 2:
        tp, tm, dE = _classes2(m)
    else:
        tp, tm, dE = torch.empty_like(m), torch.empty_like(m), torch.empty_like(m[0])
        for a in range(0, m.shape[1], 1 << 17):
            U, S, Vh = torch.linalg.svd(m[:, a:a + (1 << 17)].T.reshape(-1, 3, 3))
            Q = U @ Vh
            o = Q - 2 * U[:, :, 2:] @ Vh[:, 2:, :]
            up = (torch.linalg.det(Q) > 0)[:, None, None]
            tp[:, a:a + (1 << 17)] = torch.where(up, Q, o).reshape(-1, 9).T
            tm[:, a:a + (1 << 17)] = torch.where(up, o, Q).reshape(-1, 9).T
            dE[a:a + (1 << 17)] = torch.where(up[:, 0, 0], 2 * S[:, 2], -2 * S[:, 2])
    order = torch.sort(dE, descending=True, stable=True).indices
    sel = torch.zeros(dE.numel(), dtype=torch.bool, device="cuda")
    sel[order[:n_plus]] = True
    return torch.where(sel, tp, tm).view((n * n,) + dims)
