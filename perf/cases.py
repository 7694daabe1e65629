"""The work that users of the library have it do, as cases to be timed and compared.

A case is one call of the public entry points (a render of a batch of pose cells, of one pose box
through a partition, concrete renders at sampled poses) on a seeded synthetic scene.  Sizes are the
ones of ``synth.py``'s workloads and serving mix, and generic ones between them.

Every render names its tile edge: with tile = 0 the library times candidates on the first call, and
two runs could then choose different ones, whose bounds differ by the early stop's 2e-5.  The edges
here are the ones its autotuner chooses for these sizes (8 for the small scenes, else 16).
"""
import math

import numpy as np
import torch

from paper_2503_00308_gb300 import ar, synth

# pose dimensions that move: x translation only (1 pose variable), translation and yaw (4), all (6)
MOVES = {"x": (1, 0, 0, 0, 0, 0), "xyz_yaw": (1, 1, 1, 0, 1, 0), "6dof": (1, 1, 1, 1, 1, 1)}


def _case(name, kind, scene, n, width, height, move, splits, half_t, half_deg, scale=1.0, tile=16, **more):
    c = {"kind": kind, "scene": scene, "n": n, "width": width, "height": height, "move": move, "splits": splits,
         "half_t": half_t, "half_deg": half_deg, "scale": scale, "tile": tile, **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: the check scene, one translation cell (latency and launches)
        _case("tiny64", "abstract", "cube", 64, 32, 32, "x", "1x1x1x1x1x1", 0.01, 0.0),
        # a control loop that may not allocate: a small scene, two narrow cells, fixed scratch
        _case("noalloc3k", "noalloc", "object", 3000, 161, 119, "6dof", "2x1x1x1x1x1", 0.02, 0.5, scale=0.05),
        # the smallest serving request: one cell of the 10k scene
        _case("query10k", "abstract", "object", 10_000, 200, 200, "6dof", "1x1x1x1x1x1", 0.02, 0.5, tile=8),
        # the 10k object workload: 16 cells, 4 pose variables
        _case("object10k", "abstract", "object", 10_000, 200, 200, "xyz_yaw", "2x2x2x1x2x1", 0.05, 1.0, tile=8),
        # one pose box through a uniform partition, joined on the device
        _case("partition10k", "partition", "object", 10_000, 400, 300, "xyz_yaw", "4x2x2x1x2x1", 0.05, 1.0),
        # one pose box refined adaptively: a series of small dependent renders
        _case("refine10k", "refine", "object", 10_000, 200, 200, "6dof", "1x1x1x1x1x1", 0.02, 0.5, tile=8, rounds=5),
        # a set of scenes (parameter boxes) under the relational blend, odd image and cell counts
        _case("boxes50k", "relational", "object", 50_000, 403, 301, "6dof", "3x1x1x1x2x1", 0.02, 0.5, scale=0.05,
              boxes=True),
        # one cell of the 300k scene at the largest resolution (a large single query)
        _case("query300k", "abstract", "object", 300_000, 1280, 720, "6dof", "1x1x1x1x1x1", 0.02, 0.5),
        # the headline workload: 300k Gaussians, 64 cells
        _case("object300k", "abstract", "object", 300_000, 800, 800, "6dof", "2x2x2x2x2x2", 0.02, 0.5),
        # the same scene under narrow cells, whose bounds are informative: deep sweeps
        _case("fine300k", "abstract", "object", 300_000, 800, 800, "6dof", "2x2x2x1x2x1", 0.02, 0.5, scale=0.05),
        # a camera inside a large scene, the centres of 16 cells (the whole cells' bounds are all 0 and 1)
        _case("unbounded750k", "abstract", "box", 750_000, 1280, 720, "6dof", "2x2x2x1x2x1", 0.10, 2.0, scale=0.1),
        # concrete renders at sampled poses (the soundness check of the 300k scene)
        _case("concrete300k", "concrete", "object", 300_000, 800, 800, "6dof", "1x1x1x1x1x1", 0.02, 0.5, poses=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(["abstract", "relational", "noalloc", "partition", "refine", "concrete"], [8, 2, 1, 2, 1, 2])[0]
    scene = "box" if kind == "abstract" and rng.random() < 0.2 else "object"
    small = kind in ("noalloc", "refine")
    n = int(_log(rng, 64, 3000 if kind == "noalloc" else 20_000 if small else 750_000 if scene == "box" else 300_000))
    w = int(_log(rng, 32, 200 if small else 1280))
    h = max(8, min(800, int(w * rng.uniform(0.5, 1.0))))
    move = rng.choice(["x", "xyz_yaw", "6dof", "6dof"])
    # cells: within a sixth of the largest listed call's pixel-cells (narrow cells sweep deep)
    most = {"noalloc": 2, "refine": 1, "concrete": 1}.get(kind, 64)
    most = max(1, min(most, int(6e6 / (w * h)), int(12e6 / n)))
    sp = [1] * 6
    for k in rng.sample(range(6), 6):
        if MOVES[move][k]:
            top = min(4, most // math.prod(sp))
            sp[k] = rng.randint(1, top) if top > 1 else 1
    scale = _log(rng, 0.05, 0.2) if scene == "box" else _log(rng, 0.05, 1.0)
    t, deg = (0.10, 2.0) if scene == "box" else (0.02, 0.5)
    more = {"refine": {"rounds": rng.randint(1, 5)}, "concrete": {"poses": rng.randint(1, 3)}}.get(kind, {})
    if kind in ("abstract", "relational") and scene == "object" and rng.random() < 0.2:
        more["boxes"] = True
    tile = 8 if n <= 20_000 and kind != "noalloc" and rng.random() < 0.7 else 16
    return _case(None, kind, scene, n, w, h, move, "x".join(map(str, sp)), t, deg, scale, tile, **more)


def _inputs(case, seed):
    """Scene, camera and pose cells of a case: lo, hi [n_cells, 6]; the whole box for the partition kinds."""
    n, w, h = case["n"], case["width"], case["height"]
    if case["scene"] == "cube":
        sc, cam = synth.cube_scene(n, seed), synth.look_camera(w, h, float(w), centre=(0.0, 0.0, -3.0))
    elif case["scene"] == "object":
        sc, cam = synth.object_scene(n, seed), synth.look_camera(w, h, (1.1 if n <= 20_000 else 1.375) * w)
    else:
        sc, cam = synth.box_scene(n, seed), synth.look_camera(w, h, 0.703 * w, centre=(0.0, 0.0, 0.0))
    on = np.array(MOVES[case["move"]])
    half = on * np.array([case["half_t"]] * 3 + [case["half_deg"] * synth.DEG] * 3)
    splits = [int(s) for s in case["splits"].split("x")]
    one = case["kind"] in ("partition", "refine", "concrete")
    lo, hi = synth.cell_grid(half, [1] * 6 if one else splits)
    mid, rad = 0.5 * (lo + hi), 0.5 * (hi - lo) * case["scale"]
    return sc, cam, mid - rad, mid + rad, splits


def prepare(case, seed):
    sc, cam, lo, hi, splits = _inputs(case, seed)
    s = {"case": case, "camera": cam, "lo": lo, "hi": hi, "scene": ar.Scene(sc)}
    kind, shape = case["kind"], (cam.height, cam.width, 3)
    if kind == "relational":
        ar.ar_scene_set_blend(s["scene"].handle, ar.AR_BLEND_RELATIONAL)
    if case.get("boxes"):
        s["scene"].set_boxes(synth.scene_boxes(sc, seed + 1, mean_d=(0.002, 0.0, 0.001), opacity_scale=0.9,
                                               opacity_add=0.05, red_add=0.1))
    # the marshalled arguments of the ar_* calls without a Scene method
    s["intr"], s["pose"], s["cells"] = ar.make_intrinsics(cam), ar.make_pose(cam), ar.make_cells(lo, hi)
    if kind == "concrete":
        s["deltas"] = synth.sample_poses(np.random.default_rng(seed + 2), lo[0], hi[0], case["poses"])
        s["out"] = torch.zeros((case["poses"],) + shape, dtype=torch.float32, device="cuda")
    else:
        if kind in ("partition", "refine"):
            s["parts"] = splits
        else:
            shape = (lo.shape[0],) + shape
        s["out"] = [torch.zeros(shape, dtype=torch.float32, device="cuda") for _ in range(2)]
    return s


def run(s):
    case, scene, out = s["case"], s["scene"], s["out"]
    kind, tile = case["kind"], case["tile"]
    if kind == "concrete":
        scene.render_concrete(s["camera"], s["deltas"], out)
    elif kind == "noalloc":
        ar.ar_render_abstract_noalloc(scene.handle, s["intr"], s["pose"], s["cells"], len(s["cells"]), tile, *out)
    elif kind == "partition":
        ar.ar_render_abstract_partitioned(scene.handle, s["intr"], s["pose"], s["cells"][0], s["parts"], tile, *out)
    elif kind == "refine":
        lo, hi = ar.ar_render_abstract_refined(scene.handle, s["intr"], s["pose"], s["cells"][0], case["rounds"], tile,
                                               *out)
        return out + [lo, hi]  # and the pieces it ended with
    else:
        scene.render(s["camera"], s["lo"], s["hi"], *out, tile=tile)
    return out


def work(case):
    """Scene read once (56 B per Gaussian), bounds written once; per (Gaussian, cell) pair the depth chain
    (about 130 operations), per pixel and cell one opacity relaxation (58 M + 283) at the least: how many a
    pixel needs depends on the scene, and is several dozen more where its bounds are informative."""
    n, px, kind = case["n"], case["width"] * case["height"], case["kind"]
    cells = math.prod(int(s) for s in case["splits"].split("x"))
    if kind == "refine":  # 1, 2, 3, 5, 8, ... pieces in turn
        cells, p = 1, 1
        for _ in range(case["rounds"]):
            p += (p + 1) // 2
            cells += p
    if kind == "concrete":
        return {"bytes": 56 * n + 12 * px * case["poses"], "flops": case["poses"] * (n * 150 + px * 30)}
    images = 1 if kind in ("partition", "refine") else cells
    per_pixel = 58 * {"x": 1, "xyz_yaw": 4, "6dof": 6}[case["move"]] + 283
    return {"bytes": 56 * n + 24 * px * images, "flops": cells * (n * 130 + px * per_pixel)}


# ------------------------------------------------------------------ the same numbers in 64 bits
# A bounded scalar over p in [-1, 1]^M is (c, lo, hi): c . p + lo <= v <= c . p + hi, c [..., M].

def _conc(x):
    r = x[0].abs().sum(-1)
    return x[1] - r, x[2] + r


def _lin(*terms):
    """sum of a x over pairs (a, x)"""
    c = lo = hi = 0.0
    for a, x in terms:
        a = torch.as_tensor(a, dtype=torch.float64, device=x[1].device)
        pos = a >= 0
        c = c + a[..., None] * x[0]
        lo = lo + a * torch.where(pos, x[1], x[2])
        hi = hi + a * torch.where(pos, x[2], x[1])
    return c, lo, hi


def _shift(x, lo, hi):
    return x[0], x[1] + lo, x[2] + hi


def _mul(x, y):
    """averaged McCormick planes"""
    (xl, xh), (yl, yh) = _conc(x), _conc(y)
    z = _lin((0.5 * (yl + yh), x), (0.5 * (xl + xh), y))
    return _shift(z, -0.5 * (xl * yl + xh * yh), -0.5 * (xh * yl + xl * yh))


def _sqr(x):
    """tangent at the midpoint below, secant above"""
    xl, xh = _conc(x)
    s = xl + xh
    return _shift(_lin((s, x)), -0.25 * s * s, torch.maximum(xl * xl - s * xl, xh * xh - s * xh))


def _sum(*xs):
    return _lin(*[(1.0, x) for x in xs])


def _imul(a, b):
    p = torch.stack(torch.broadcast_tensors(a[0] * b[0], a[0] * b[1], a[1] * b[0], a[1] * b[1]))
    return p.amin(0), p.amax(0)


def _iadd(*xs):
    return sum(x[0] for x in xs), sum(x[1] for x in xs)


def _scene64(sc, dev):
    t = lambda a: torch.as_tensor(np.asarray(a), device=dev).double()  # noqa: E731
    q = t(sc.quat)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    o = t(sc.opacity)
    return t(sc.uw), R * t(sc.logscale).exp()[:, None, :], o, 2 * (255 * o).log(), t(sc.rgb)


def _rot(axis, a):
    """rotation about an axis and its derivative"""
    c, s = math.cos(a), math.sin(a)
    R, D = np.zeros((3, 3)), np.zeros((3, 3))
    i, j = [(1, 2), (2, 0), (0, 1)][axis]
    R[axis, axis] = 1.0
    R[i, i] = R[j, j] = c
    R[i, j], R[j, i] = -s, s
    D[i, i] = D[j, j] = -s
    D[i, j], D[j, i] = -c, c
    return R, D


def _rotations(th):
    (X, dX), (Y, dY), (Z, dZ) = (_rot(k, th[k]) for k in range(3))
    return X @ Y @ Z, [dX @ Y @ Z, X @ dY @ Z, X @ Y @ dZ]


def _concrete64(sc, cam, delta, dev):
    """GSplat at one pose, Gaussians blended front to back."""
    uw, Mw, o, tau, rgb = _scene64(sc, dev)
    R = torch.as_tensor(_rotations(delta[3:])[0].T @ cam.R_wc, device=dev)
    uc = (uw - torch.as_tensor(cam.t + delta[:3], device=dev)) @ R.T
    Mc, d = R @ Mw, uc[:, 2]
    Mp = torch.stack([cam.fx * (d[:, None] * Mc[:, 0] - uc[:, :1] * Mc[:, 2]),
                      cam.fy * (d[:, None] * Mc[:, 1] - uc[:, 1:2] * Mc[:, 2])], 1)
    X = Mp @ Mp.transpose(1, 2)
    det = X[:, 0, 0] * X[:, 1, 1] - X[:, 0, 1] ** 2
    mu = torch.stack([cam.cx + cam.fx * uc[:, 0] / d, cam.cy + cam.fy * uc[:, 1] / d], 1)
    off = (mu - torch.tensor([cam.cx, cam.cy], device=dev)).abs()
    keep = (d > cam.near) & (det > 0) & (tau >= 0) & (off[:, 0] <= 0.65 * cam.width) & (off[:, 1] <= 0.65 * cam.height)
    at = keep.nonzero()[:, 0]
    at = at[d[at].argsort()]
    d, mu, X, det, o, tau, rgb = d[at], mu[at], X[at], det[at], o[at], tau[at], rgb[at]
    rx, ry = (tau * X[:, 0, 0]).sqrt() / d ** 2, (tau * X[:, 1, 1]).sqrt() / d ** 2
    out = torch.zeros((cam.height, cam.width, 3), dtype=torch.float64, device=dev)
    T0, T1 = 32, 64  # blocks of pixels, each over the Gaussians that reach it
    for y0 in range(0, cam.height, T0):
        for x0 in range(0, cam.width, T1):
            y = torch.arange(y0, min(y0 + T0, cam.height), device=dev) + 0.5
            x = torch.arange(x0, min(x0 + T1, cam.width), device=dev) + 0.5
            g = ((mu[:, 1] + ry >= y[0] - 1) & (mu[:, 1] - ry <= y[-1] + 1) & (mu[:, 0] + rx >= x[0] - 1)
                 & (mu[:, 0] - rx <= x[-1] + 1)).nonzero()[:, 0]
            T = torch.ones((len(y), len(x)), dtype=torch.float64, device=dev)
            for b in g.split(512) if len(g) else ():  # front to back
                dx, dy = x[None, :, None] - mu[b, 0], y[:, None, None] - mu[b, 1]
                m = d[b] ** 4 * (X[b, 1, 1] * dx * dx - 2 * X[b, 0, 1] * dx * dy + X[b, 0, 0] * dy * dy) / det[b]
                a = torch.where(m <= tau[b], o[b] * (-0.5 * m).exp(), 0.0)
                P = (1 - a).cumprod(-1)
                before = torch.cat([torch.ones_like(P[..., :1]), P[..., :-1]], -1)
                out[y0:y0 + T0, x0:x0 + T1] += T[..., None] * ((before * a) @ rgb[b])
                T = T * P[..., -1]
                if float(T.max()) < 1e-13:
                    break
    return out.clamp(0, 1)


def _abstract64(sc, cam, lo, hi, slots, dev):
    """AbstractSplat on one cell: lower and upper images, or None where MatrixInv would need a divided cell."""
    uw, Mw, o, tau, rgb = _scene64(sc, dev)
    n, M = uw.shape[0], max(1, len(slots))
    ctr, h = 0.5 * (lo + hi), 0.5 * (hi - lo)
    f = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
    R, dR = _rotations(ctr[3:])
    rem = 0.5 * h[3:].sum() ** 2

    def form(c, k, r=0.0):
        v = torch.zeros(M, dtype=torch.float64, device=dev)
        for j, s in enumerate(slots):
            v[j] = c[s]
        return v, f(k - r), f(k + r)

    R0 = np.asarray(cam.R_wc)
    Rf = [[form([0, 0, 0] + [dR[k][i, j] * h[3 + k] for k in range(3)], R[i, j], rem) for j in range(3)] for i in range(3)]
    sf = [form([R0[a, k] * h[k] for k in range(3)] + [0] * 3, float(R0[a] @ ctr[:3])) for a in range(3)]
    g = form([-float(R[:, 2] @ R0[:, k]) * h[k] for k in range(3)] + [0] * 3, 0.0)
    v, N = (uw - f(cam.t)) @ f(R0).T, f(R0) @ Mw
    vs = [_shift(_lin((-1.0, sf[b])), v[:, b], v[:, b]) for b in range(3)]
    uc = [_sum(*[_mul(Rf[b][a], vs[b]) for b in range(3)]) for a in range(3)]
    d = uc[2]
    dlo, dhi = _conc(d)
    klo, khi = _conc((d[0] - g[0], d[1], d[2]))
    pad = 1e-9 * (1 + torch.maximum(klo.abs(), khi.abs()))
    klo, khi = klo - pad, khi + pad
    # pixel boxes from intervals
    Ri = [[tuple(_conc(Rf[i][j])) for j in range(3)] for i in range(3)]
    vi = [_conc(x) for x in vs]
    D = dlo.clamp(min=cam.near), dhi
    uci = [_iadd(*[_imul(Ri[b][a], vi[b]) for b in range(3)]) for a in range(2)]
    fc, cc, size = (cam.fx, cam.fy), (cam.cx, cam.cy), (cam.width, cam.height)
    keep, inside, box = (dhi > cam.near) & (tau >= 0), torch.ones(n, dtype=torch.bool, device=dev), []
    for a in range(2):
        q = _imul(uci[a], (1 / D[1], 1 / D[0]))
        mu = cc[a] + fc[a] * q[0], cc[a] + fc[a] * q[1]
        ml, mh = mu[0] - 1e-9 * (1 + mu[0].abs()), mu[1] + 1e-9 * (1 + mu[1].abs())
        keep = keep & (ml <= cc[a] + 0.65 * size[a]) & (mh >= cc[a] - 0.65 * size[a])
        inside = inside & (ml >= cc[a] - 0.65 * size[a]) & (mh <= cc[a] + 0.65 * size[a])
        Xr = 0.0
        for c in range(3):
            m = [_iadd(*[_imul(Ri[b][k], (N[:, b, c], N[:, b, c])) for b in range(3)]) for k in range(3)]
            p, u = _imul(D, m[a]), _imul(uci[a], m[2])
            p = fc[a] * (p[0] - u[1]), fc[a] * (p[1] - u[0])
            Xr = Xr + torch.maximum(p[0] ** 2, p[1] ** 2)
        r = (tau.clamp(min=0) * Xr).sqrt() / D[0] ** 2
        xl, xh = mu[0] - r, mu[1] + r
        xl, xh = xl - 1e-9 * (1 + xl.abs()), xh + 1e-9 * (1 + xh.abs())
        x0, x1 = (xl - 0.5).ceil().clamp(min=0), (xh - 0.5).floor().clamp(max=size[a] - 1)
        keep = keep & (x0 <= x1)
        box.append((x0, x1))
    at = keep.nonzero()[:, 0]
    pick = lambda x: (x[0].expand(n, M)[at], x[1].expand(n)[at], x[2].expand(n)[at])  # noqa: E731
    uc, N, o, tau, rgb = [pick(x) for x in uc], N[at], o[at], tau[at], rgb[at]
    klo, khi, inside = klo[at], khi[at], inside[at] & (dlo[at] > cam.near)
    (bx0, bx1), (by0, by1) = [(b[0][at], b[1][at]) for b in box]
    d = uc[2]
    Mc = [[_lin(*[(N[:, b, c], Rf[b][a]) for b in range(3)]) for c in range(3)] for a in range(3)]
    Mp = [[_sum(_mul(_lin((fc[a], d)), Mc[a][c]), _mul(_lin((-fc[a], uc[a])), Mc[2][c])) for c in range(3)]
          for a in range(2)]
    S, P = _sqr(d), [_mul(d, _lin((fc[a], uc[a]), (cc[a], d))) for a in range(2)]
    # MatrixInv: Taylor series around the inverse of the centre matrix
    X = [_sum(*[_sqr(Mp[0][c]) for c in range(3)]), _sum(*[_mul(Mp[0][c], Mp[1][c]) for c in range(3)]),
         _sum(*[_sqr(Mp[1][c]) for c in range(3)])]
    mid = [0.5 * sum(_conc(x)) for x in X]
    det = mid[0] * mid[2] - mid[1] ** 2
    X0 = [mid[2] / det, -mid[1] / det, -mid[1] / det, mid[0] / det]
    Xf = [X[0], X[1], X[1], X[2]]
    E = [_shift(_lin((-X0[s], Xf[2 * r]), (-X0[2 + s], Xf[2 * r + 1])), float(r == s), float(r == s))
         for r in range(2) for s in range(2)]
    rho = sum(torch.maximum(*[b.abs() for b in _conc(e)]) ** 2 for e in E).sqrt()
    if not bool(((det > 0) & (rho < 1 - 2.0 ** -10)).all()):
        return None
    k = torch.full_like(rho, 8.0)
    for _ in range(16):
        k = torch.where(rho ** (k + 1) / (1 - rho) > 2.0 ** -24, k + 1, k)
    k = k.clamp(max=24)
    pw, T = E, E
    for i in range(2, int(k.max()) + 1 if len(at) else 2):
        pw = [_sum(_mul(pw[2 * r], E[s]), _mul(pw[2 * r + 1], E[2 + s])) for r in range(2) for s in range(2)]
        on = (k >= i).double()
        T = [_lin((1.0, t), (on, p)) for t, p in zip(T, pw)]
    eps = sum(x * x for x in X0).sqrt() * rho ** (k + 1) / (1 - rho)
    conic = [_shift(_lin((X0[2 * r], T[s]), (X0[2 * r + 1], T[2 + s])), X0[2 * r + s] - eps, X0[2 * r + s] + eps)
             for r in range(2) for s in range(2)]
    W = [[_sum(_mul(conic[2 * r], Mp[0][c]), _mul(conic[2 * r + 1], Mp[1][c])) for c in range(3)] for r in range(2)]
    out = [torch.zeros((cam.height, cam.width, 3), dtype=torch.float64, device=dev) for _ in range(2)]
    px = torch.arange(cam.width, device=dev)[:, None]
    for y in range(cam.height):  # a row of pixels over the Gaussians whose boxes meet it
        r = ((by0 <= y) & (by1 >= y)).nonzero()[:, 0]
        if not len(r):
            continue
        sub = lambda x: (x[0][r], x[1][r], x[2][r])  # noqa: E731
        meets = (px >= bx0[r]) & (px <= bx1[r])
        delta = []
        for a, u in ((0, px + 0.5), (1, torch.full_like(px, y) + 0.5)):
            s, p = sub(S), sub(P[a])
            delta.append((u[..., None] * s[0] - p[0], u * s[1] - p[2], u * s[2] - p[1]))
        m = _sum(*[_sqr(_sum(_mul(delta[0], sub(W[0][c])), _mul(delta[1], sub(W[1][c])))) for c in range(3)])
        L, alo, U, ahi = _opacity64(m, o[r], tau[r], inside[r], meets)
        # BlendInd: products over keys strictly below a value
        one = torch.ones_like(alo[:, :1])
        i_lo, i_hi = klo[r].argsort(), khi[r].argsort()
        before_a = torch.cat([one, (1 - ahi)[:, i_lo].cumprod(1)], 1)
        before_b = torch.cat([one, (1 - alo)[:, i_hi].cumprod(1)], 1)
        T_lo = before_a[:, torch.searchsorted(klo[r][i_lo], khi[r])] / (1 - ahi)
        T_hi = before_b[:, torch.searchsorted(khi[r][i_hi], klo[r])]
        for side, (Tr, F, sign) in enumerate(((T_lo, L, -1.0), (T_hi, U, 1.0))):
            c = torch.einsum("pg,gk,pgj->pkj", Tr, rgb[r], F[0])
            out[side][y] = (Tr * F[1]) @ rgb[r] + sign * c.abs().sum(-1)
    return out[0].clamp(0, 1), out[1].clamp(0, 1)


def _opacity64(m, o, tau, inside, meets):
    """Lower and upper forms (c, k) of the effective opacity from the bounded m, with their enclosures."""
    ml, mh = _conc(m)
    xl, xu = -0.5 * mh, torch.maximum((-0.5 * ml).clamp(max=0), -0.5 * mh)
    el, eu = xl.exp(), xu.exp()
    k1 = o * el
    L = [-0.5 * k1[..., None] * m[0], k1 * (1 - xl) - 0.5 * k1 * m[2]]
    w = xu - xl
    s = o * torch.where(w > 0, (eu - el) / torch.where(w > 0, w, 1.0), eu)
    U = [-0.5 * s[..., None] * m[0], o * el - s * xl - 0.5 * s * m[1]]
    lam = ((o * 1.25 - (U[1] + U[0].abs().sum(-1))) / (0.25 * o)).clamp(0, 1)
    ramp = (mh - ml).clamp(0, 0.5)
    safe = torch.where(ramp > 0, ramp, 1.0)
    psi2 = torch.where(ml <= tau, 0.0, torch.where(ramp > 0, ((ml - tau) / safe).clamp(0, 1), 1.0))
    psi = torch.where(mh > tau, 1.0, torch.where(ramp > 0, ((mh - tau + ramp) / safe).clamp(0, 1), 0.0))
    keep = (1 - psi2) * meets
    U = [(keep * lam)[..., None] * U[0], keep * (lam * U[1] + (1 - lam) * o)]
    L[1] = L[1] - psi / 255
    r = L[0].abs().sum(-1)
    l0, l1 = L[1] - r, L[1] + r
    mu = torch.where(l0 >= 0, 1.0, torch.where(l1 <= 0, 0.0, (l1 / torch.where(l1 > l0, l1 - l0, 1.0)).clamp(0, 1)))
    mu = mu * inside * meets
    L = [mu[..., None] * L[0], mu * L[1]]
    alo = (L[1] - L[0].abs().sum(-1)).clamp(min=0)
    return L, alo, U, torch.minimum(U[1] + U[0].abs().sum(-1), o) * meets


def exact(case, seed):
    sc, cam, lo, hi, _ = _inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    px = cam.width * cam.height
    if case["kind"] == "concrete":
        if case["n"] * px * case["poses"] > 1e12:
            return None  # more than about 20 seconds
        deltas = synth.sample_poses(np.random.default_rng(seed + 2), lo[0], hi[0], case["poses"])
        return torch.stack([_concrete64(sc, cam, d, dev) for d in deltas])
    # narrow cells only: under wide ones the lower bounds are all but zero, and so is what they are compared with
    narrow = case["scene"] == "cube" or (case["scene"] == "object" and case["scale"] <= 0.1)
    if case["kind"] not in ("abstract", "noalloc") or case.get("boxes") or not narrow:
        return None
    if case["n"] * px * len(lo) > 4e8 or cam.height * len(lo) > 400:
        return None
    slots = [k for k in range(6) if (hi[:, k] > lo[:, k]).any()]
    got = [_abstract64(sc, cam, lo[c], hi[c], slots, dev) for c in range(len(lo))]
    if any(g is None for g in got):
        return None
    return [torch.stack([g[side] for g in got]) for side in range(2)]
