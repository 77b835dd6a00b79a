"""Timed cases of the random-sampling multiscale solver, through its public entry points.

A case names a path of the package, a medium, a partition into buffered patches and the
options of the call; a seed gives the medium's random modes, the Gaussian sample stream and
the boundary data.  `exact` restates the method in 64 bits with plain torch and numpy.

Paths
  step      a new medium to its first solution: build, local solves, bases, one online solve
  sample    build and local solves, all snapshot blocks read back (what sharded runs exchange)
  extract   bases, online operators and factor from sampled snapshots, then a first solution
  online    solutions for new Dirichlet data on a prebuilt basis
  map       the same through the boundary-to-coefficient map of the serving loop
  kinetic   the slab transport example: build, sample, extract, solve
  operator  the streaming matrix-free operator on a stack of tiles
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1807_08848_gb300 as msp

F64 = torch.float64


# ------------------------------------------------------------------ the cases

def _elliptic(path, name=None, **kw):
    c = {"path": path, "medium": "lognormal", "n": 512, "eps_log2": 5, "patches": 8, "ragged": False, "buffer": 16,
         "samples": 128, "precision": "mixed", "solver": "direct", "tol": 1e-12, "tau": 1e-6, "online_tol": 1e-10,
         "batch": 1}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _kinetic(name=None, **kw):
    c = {"path": "kinetic", "n": 8192, "eps_log2": 8, "n_v": 64, "patches": 64, "buffer": 32, "samples": 96, "g": 0.5,
         "solver": "direct", "precision": "fp64", "tol": 1e-13, "tau": 1e-6}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one pass of the small example: latency and launches count
        _elliptic("step", "step_129_periodic", medium="periodic", n=128, eps_log2=4, patches=4, buffer=8, samples=40),
        # the same with plain FP64 conjugate gradients, the entry points' default precision
        _elliptic("step", "step_129_fp64", n=128, eps_log2=4, patches=4, buffer=8, samples=40, precision="fp64",
                  solver="split"),
        # uneven patches of a high-contrast medium, ragged tiles
        _elliptic("step", "step_641_channels_ragged", medium="channels", n=640, eps_log2=5, patches=11, ragged=True,
                  buffer=12, samples=96),
        # the benchmark's workload: 1024 patches, 143356 local solves
        _elliptic("step", "step_2049_lognormal", n=2048, eps_log2=7, patches=32),
        # local solves alone, the size of one serving medium and an odd ragged one
        _elliptic("sample", "sample_513_lognormal"),
        _elliptic("sample", "sample_1023_ragged", n=1022, eps_log2=6, patches=13, ragged=True, buffer=17, samples=150),
        # bases of new snapshots on a prebuilt medium
        _elliptic("extract", "extract_513_lognormal"),
        # one request, and a batch of requests, on prebuilt bases (plain FP64 iteration)
        _elliptic("online", "online_2049_single", n=2048, eps_log2=7, patches=32),
        _elliptic("online", "online_513_batch32", batch=32),
        # a served batch through the map, interactive latency
        _elliptic("map", "map_513_batch32", batch=32),
        # transport slab with Henyey-Greenstein scattering
        _kinetic("kinetic_8193_hg"),
        # operator on all tiles of one medium, larger than the cache
        _elliptic("operator", "operator_1025_fp32", n=1024, eps_log2=6, patches=16, samples=96),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    largest = max(work(c)["flops"] for c in listed())
    while True:
        path = rng.choice(["step", "step", "step", "sample", "sample", "extract", "online", "online", "map", "kinetic",
                           "operator"])
        if path == "kinetic":
            m = _log_uniform(rng, 4, 64)
            cells = _log_uniform(rng, 16, 128)
            n_v = 2 * _log_uniform(rng, 4, 32)
            return _kinetic(n=m * cells, eps_log2=rng.randint(2, 8), n_v=n_v, patches=m,
                            buffer=rng.randint(4, min(32, cells)), samples=n_v + 2 * rng.randint(0, 16),
                            g=rng.choice([0.0, 0.5, -0.3]))
        width = rng.randint(24, 72)                       # cells per patch, about
        top = {"step": 2048, "sample": 1100, "extract": 1100, "online": 2048, "map": 520, "operator": 1100}[path]
        n = _log_uniform(rng, 96, top)
        m = max(2, n // width)
        buffer = rng.randint(4, min(20, width // 2))
        medium = rng.choice(["lognormal", "lognormal", "channels", "periodic"])
        kw = {}
        if path in ("online", "map"):
            kw["batch"] = rng.choice([1, 1, 2, 5, 8, 17, 32]) if n <= 1100 else 1
            medium = "lognormal"
        if path == "operator":
            kw["precision"] = rng.choice(["mixed", "mixed", "fp64"])
            kw["samples"] = rng.randint(8, 96)
        else:
            kw["samples"] = rng.randint(40, 160)
            if path in ("step", "sample") and n <= 160 and rng.random() < 0.3:
                kw.update(precision="fp64", solver="split")
        c = _elliptic(path, medium=medium, n=n, eps_log2=max(3, int(math.log2(n)) - 4), patches=m, ragged=True,
                      buffer=buffer, **kw)
        if work(c)["flops"] <= largest:
            return c


# ------------------------------------------------------------------ inputs

def _breaks(case):
    n, m = case["n"], case["patches"]
    if not case["ragged"]:
        assert n % m == 0
        return (np.arange(m + 1, dtype=np.int32) * (n // m),) * 2
    out = []
    for axis in (0, 1):                                   # widths within a quarter of the mean
        r = np.random.default_rng([n, m, axis])
        b = np.arange(m + 1) * (n / m)
        b[1:-1] += r.uniform(-0.12, 0.12, m - 1) * (n / m)
        out.append(np.rint(b).astype(np.int32))
    return tuple(out)


def _medium_spec(case, seed):
    r = np.random.default_rng([seed, 1])
    eps = 2.0 ** -case["eps_log2"]
    s = SimpleNamespace(kind=0, n_cells=case["n"], eps=eps, modes=np.zeros((0, 4)), amp=0.5, norm=1.0,
                        channels=np.zeros((0, 3)), width=0.0, contrast=1.0, user_aE=None, user_aN=None)
    if case["medium"] == "lognormal":                     # 64 random Fourier modes, 1 <= |k| <= 1 / eps
        s.kind, s.norm = 1, 1.0 / 8.0
        rad, ang = np.sqrt(r.uniform(1.0, (1.0 / eps) ** 2, 64)), r.uniform(0.0, 2.0 * np.pi, 64)
        k = np.trunc(np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1))
        k[(k == 0).all(1)] = 1.0
        s.modes = np.concatenate([k, r.standard_normal((64, 2))], 1)
    elif case["medium"] == "channels":                    # 8 strips of width eps, contrast 1000
        s.kind, s.width, s.contrast = 2, eps, 1e3
        s.channels = np.concatenate([r.uniform(0, 1, (8, 2)), r.uniform(0, math.pi, (8, 1))], 1)
    return s


def _patch_spec(case):
    xb, yb = _breaks(case)
    n = (len(xb) - 1) * (len(yb) - 1)
    return SimpleNamespace(x_breaks=xb, y_breaks=yb, buffers=np.full(n, case["buffer"], np.int32),
                           samples=np.full(n, case["samples"], np.int32))


def _ring(X0, X1, Y0, Y1):
    """Nodes (i, j) of a box's ring, counter-clockwise from its lower left corner."""
    a, b = np.arange(X0, X1), np.arange(Y0, Y1)
    i = np.concatenate([a, np.full(len(b), X1), a[::-1] + 1, np.full(len(b), X0)])
    j = np.concatenate([np.full(len(a), Y0), b, np.full(len(a), Y1), b[::-1] + 1])
    return i, j


def _phi(case, seed):
    """Dirichlet data: 16 random Fourier modes with |k| <= 8 per data set."""
    r = np.random.default_rng([seed, 2])
    i, j = _ring(0, case["n"], 0, case["n"])
    k = r.integers(-8, 9, (case["batch"], 16, 2))
    a = r.standard_normal((case["batch"], 16, 2)) / 4.0
    ph = 2.0 * np.pi / case["n"] * (k[..., 0:1] * i + k[..., 1:2] * j)
    return (a[..., 0:1] * np.cos(ph) + a[..., 1:2] * np.sin(ph)).sum(1)


def _medium(case, s):
    med = msp.Medium(s.medium, s.partition)
    if case["precision"] == "mixed":
        med.set_launch("mixed", case["solver"])
    return med


def _sample(case, s, med):
    med.sample(s.seed, case["precision"], tol=case["tol"], max_iter=20000)


def prepare(case, seed):
    s = SimpleNamespace(case=case, seed=seed)
    if case["path"] == "kinetic":
        r = np.random.default_rng([seed, 3])
        s.inflow = torch.from_numpy(2.0 + r.standard_normal((1, 2, case["n_v"]))).cuda()
        return s
    s.medium, s.partition = _medium_spec(case, seed), _patch_spec(case)
    if case["path"] == "operator":
        s.med = msp.Medium(s.medium, s.partition)
        rows, cols = s.med.tile_shape()
        g = torch.Generator(device="cuda").manual_seed(seed)
        s.x = torch.randn((s.med.n_patches, case["samples"], rows, (cols + 3) // 4 * 4), generator=g, device="cuda",
                          dtype=F64 if case["precision"] == "fp64" else torch.float32)
        return s
    s.phi = torch.from_numpy(_phi(case, seed)).cuda()
    if case["path"] in ("extract", "online", "map"):
        s.med = _medium(case, s)
        _sample(case, s, s.med)
    if case["path"] in ("online", "map"):
        s.basis = s.med.extract(case["tau"], case["precision"])
        s.med = None                                      # a server keeps the basis only
    if case["path"] == "map":
        s.basis.build_map()
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    case = s.case
    path = case["path"]
    if path == "kinetic":
        km = msp.KineticMedium(case["n"], 2.0 ** -case["eps_log2"], case["n_v"], case["patches"], case["buffer"],
                               case["samples"], g=case["g"])
        km.set_solver(case["solver"])
        km.sample(s.seed, tol=case["tol"], max_iter=16, precision=case["precision"])
        b = km.extract(case["tau"])
        return {"f": b.solve(s.inflow), "sigma": np.concatenate([b.sigma(m) for m in range(km.n_patches)]),
                "k": np.array([b.k(m) for m in range(km.n_patches)])}
    if path == "operator":
        return s.med.apply_operator(s.x, case["precision"])
    if path == "map":
        return s.basis.solve_map(s.phi)
    if path == "online":
        return s.basis.solve(s.phi, tol=case["online_tol"], max_iter=1000)[0]
    if path == "extract":
        med = s.med
    else:
        med = _medium(case, s)
        _sample(case, s, med)
    if path == "sample":
        s.med = med                                       # read back below, so it stays
        return torch.cat([med.snapshots(m).T.reshape(-1) for m in range(med.n_patches)])
    basis = med.extract(case["tau"], case["precision"])
    u, _ = basis.solve(s.phi, tol=case["online_tol"], max_iter=1000)
    return {"u": u, "sigma": np.concatenate([basis.sigma(m) for m in range(basis.n_patches)]),
            "k": np.array([basis.k(m) for m in range(basis.n_patches)])}


# ------------------------------------------------------------------ what a pass cannot do without

def _boxes(case):
    """Per patch (x0, x1, y0, y1) of K_m and (X0, X1, Y0, Y1) of its buffered box, columns in all, deltas."""
    n, b = case["n"], case["buffer"]
    xb, yb = (list(map(int, v)) for v in _breaks(case))
    out = []
    for q in range(len(yb) - 1):
        for p in range(len(xb) - 1):
            k = (xb[p], xb[p + 1], yb[q], yb[q + 1])
            X = (max(0, k[0] - b), min(n, k[1] + b), max(0, k[2] - b), min(n, k[3] + b))
            i, j = _ring(*X)
            on = np.nonzero((i == 0) | (i == n) | (j == 0) | (j == n))[0]
            out.append(SimpleNamespace(K=k, X=X, on=on, ring=(i, j), cols=case["samples"] + len(on),
                                       n_k=(k[1] - k[0] + 1) * (k[3] - k[2] + 1)))
    return out


def work(case):
    """Bytes: inputs and outputs of the call, each once.  Flops: of the dense parts -- block
    elimination and sweeps of the local problems over their grid rows, Householder QR and SVD of
    the snapshot blocks, and the sparse Cholesky of the normal equations by nested dissection
    (about 10 times the cube of its top separator)."""
    if case["path"] == "kinetic":
        n, v = case["n"], case["n_v"]
        nodes = n + 2 * case["patches"] * case["buffer"]
        rows = (n // case["patches"] + 1) * v
        return {"bytes": 8 * (n + 1) * v,
                "flops": nodes * (2 * v ** 3 + 4 * v * v * case["samples"]) +
                case["patches"] * (2 * rows * case["samples"] ** 2 + 20 * case["samples"] ** 3)}
    boxes = _boxes(case)
    n, B = case["n"], case["batch"]
    field = 8 * B * (n + 1) ** 2
    if case["path"] == "operator":
        es = 8 if case["precision"] == "fp64" else 4
        nodes = sum((p.X[1] - p.X[0] + 1) * (p.X[3] - p.X[2] + 1) for p in boxes)
        return {"bytes": 2 * es * nodes * case["samples"] + 2 * es * nodes, "flops": 9 * nodes * case["samples"]}
    local = qr = snaps = 0
    for p in boxes:
        nx, ny = p.X[1] - p.X[0] - 1, p.X[3] - p.X[2] - 1
        local += ny * (2 * nx ** 3 + 4 * nx * nx * p.cols)
        qr += 4 * p.n_k * p.cols ** 2 + 20 * p.cols ** 3
        snaps += 8 * p.n_k * p.cols
    unknowns = 0.55 * sum(p.cols for p in boxes)
    factor = 10 * (unknowns / len(boxes) * case["patches"]) ** 3
    if case["path"] == "sample":
        return {"bytes": snaps, "flops": local}
    if case["path"] == "step":
        return {"bytes": field, "flops": local + qr + factor}
    if case["path"] == "extract":
        return {"bytes": snaps + field, "flops": qr + factor}
    basis = 8 * sum(0.55 * p.cols * p.n_k for p in boxes)
    if case["path"] == "map":
        return {"bytes": 4 * unknowns * 4 * n + basis / 2 + field, "flops": 2 * B * unknowns * 4 * n}
    return {"bytes": basis + field, "flops": 2 * B * (basis / 8 + unknowns ** 1.5)}


# ------------------------------------------------------------------ the method in 64 bits

def _normals(seed, patch, n_nodes, n_samples, tag):
    """N(0, 1) values (n_nodes, n_samples): Philox4x32-10 counters (node pair, sample, patch, tag), Box-Muller."""
    q = np.arange((n_nodes + 1) // 2, dtype=np.uint64)[:, None]
    s = np.arange(n_samples, dtype=np.uint64)[None, :]
    lo = np.uint64(0xFFFFFFFF)
    sh = np.uint64(32)
    c = [v + np.zeros((len(q), n_samples), np.uint64) for v in (q, s, np.uint64(patch), np.uint64(tag))]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> sh) ^ c[1] ^ np.uint64(k0), b & lo, (a >> sh) ^ c[3] ^ np.uint64(k1), a & lo]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u1 = ((((c[1] << sh) | c[0]) >> np.uint64(11)).astype(np.float64) + 1.0) * 2.0 ** -53
    u2 = (((c[3] << sh) | c[2]) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
    r = np.sqrt(-2.0 * np.log(u1))
    return np.stack([r * np.cos(2 * np.pi * u2), r * np.sin(2 * np.pi * u2)], 1).reshape(-1, n_samples)[:n_nodes]


def _faces(case, spec):
    n = case["n"]
    h = 1.0 / n
    node, mid = torch.arange(n + 1, dtype=F64, device="cuda") * h, (torch.arange(n, dtype=F64, device="cuda") + 0.5) * h

    def at(x, y):
        x, y = x[None, :], y[:, None]
        if spec.kind == 0:
            return 2.0 + torch.sin(2 * math.pi * x / spec.eps) * torch.sin(2 * math.pi * y / spec.eps)
        if spec.kind == 1:
            g = torch.zeros((y.shape[0], x.shape[1]), dtype=F64, device="cuda")
            for kx, ky, a, b in spec.modes.tolist():
                ph = 2 * math.pi * (kx * x + ky * y)
                g += a * torch.cos(ph) + b * torch.sin(ph)
            return torch.exp(spec.amp * spec.norm * g)
        inside = torch.zeros((y.shape[0], x.shape[1]), dtype=torch.bool, device="cuda")
        for px, py, th in spec.channels.tolist():
            inside |= (-(x - px) * math.sin(th) + (y - py) * math.cos(th)).abs() <= 0.5 * spec.width
        return torch.where(inside, spec.contrast, 1.0).to(F64)

    return at(mid, node), at(node, mid)


def _snapshots(case, seed, boxes, aE, aN):
    """Snapshot blocks (n_k, cols): block elimination over the grid rows of groups of padded
    boxes, refined twice."""
    out = []
    for g0 in range(0, len(boxes), 32):
        grp = boxes[g0:g0 + 32]
        G = len(grp)
        nx = max(p.X[1] - p.X[0] - 1 for p in grp)
        ny = max(p.X[3] - p.X[2] - 1 for p in grp)
        nc = max(p.cols for p in grp)
        E = torch.zeros((G, ny, nx + 1), dtype=F64, device="cuda")
        Nf = torch.zeros((G, ny + 1, nx), dtype=F64, device="cuda")
        D = torch.ones((G, ny, nx), dtype=F64, device="cuda")
        U = torch.zeros((G, ny + 2, nx + 2, nc), dtype=F64, device="cuda")
        live = torch.zeros((G, ny, nx, 1), dtype=F64, device="cuda")
        for a, p in enumerate(grp):
            X0, X1, Y0, Y1 = p.X
            w, h = X1 - X0 - 1, Y1 - Y0 - 1
            E[a, :h, :w + 1] = aE[Y0 + 1:Y1, X0:X1]
            Nf[a, :h + 1, :w] = aN[Y0:Y1, X0 + 1:X1]
            D[a, :h, :w] = E[a, :h, :w] + E[a, :h, 1:w + 1] + Nf[a, :h, :w] + Nf[a, 1:h + 1, :w]
            live[a, :h, :w] = 1.0
            i, j = p.ring
            v = np.zeros((len(i), nc))
            v[:, :case["samples"]] = _normals(seed, g0 + a, len(i), case["samples"], 0x4D535045)
            v[p.on, case["samples"] + np.arange(len(p.on))] = 1.0
            U[a, torch.from_numpy(j - Y0).cuda(), torch.from_numpy(i - X0).cuda()] = torch.from_numpy(v).cuda()
        # couplings inside the boxes only
        Ei = E[:, :, 1:-1] * live[:, :, 1:, 0] * live[:, :, :-1, 0]
        Ni = Nf[:, 1:-1] * live[:, 1:, :, 0] * live[:, :-1, :, 0]
        Z, prev = [], None
        for r in range(ny):
            T = torch.diag_embed(D[:, r]) - torch.diag_embed(Ei[:, r], 1) - torch.diag_embed(Ei[:, r], -1)
            if r:
                T -= Ni[:, r - 1, :, None] * prev * Ni[:, r - 1, None, :]
            prev = torch.linalg.inv(T)
            Z.append(prev)
        for _ in range(3):
            c = U[:, 1:-1, 1:-1]
            R = (E[:, :, 1:, None] * (U[:, 1:-1, 2:] - c) + E[:, :, :-1, None] * (U[:, 1:-1, :-2] - c) +
                 Nf[:, 1:, :, None] * (U[:, 2:, 1:-1] - c) + Nf[:, :-1, :, None] * (U[:, :-2, 1:-1] - c)) * live
            w = []
            for r in range(ny):
                w.append(Z[r] @ (R[:, r] + Ni[:, r - 1, :, None] * w[-1] if r else R[:, r]))
            d = w[-1]
            U[:, ny, 1:-1] += d
            for r in range(ny - 2, -1, -1):
                d = w[r] + Z[r] @ (Ni[:, r, :, None] * d)
                U[:, r + 1, 1:-1] += d
        for a, p in enumerate(grp):
            (x0, x1, y0, y1), (X0, _, Y0, _) = p.K, p.X
            out.append(U[a, y0 - Y0:y1 - Y0 + 1, x0 - X0:x1 - X0 + 1, :p.cols].reshape(-1, p.cols).clone())
    return out


def _bases(snaps, tau):
    Q, S = [], []
    for R in snaps:
        q, t = torch.linalg.qr(R)
        u, s, _ = np.linalg.svd(t.cpu().numpy())
        k = int((s > tau * s[0]).sum())
        Q.append((q @ torch.from_numpy(u[:, :k].copy()).cuda()).cpu().numpy())
        S.append(s)
    return Q, S


def _glue(case, boxes, aE, aN, Q, phi):
    """Least squares over the skeleton: boundary values, value continuity against the first
    patch of a node, zero sum of the one-sided fluxes; then the average of the patches."""
    n = case["n"]
    aE, aN = aE.cpu().numpy(), aN.cpu().numpy()
    xb, yb = _breaks(case)
    bx, by = set(map(int, xb[1:-1])), set(map(int, yb[1:-1]))
    off = np.concatenate([[0], np.cumsum([q.shape[1] for q in Q])])
    ri, rj = _ring(0, n, 0, n)
    pos = {(int(i), int(j)): t for t, (i, j) in enumerate(zip(ri, rj))}
    held = {}
    for m, p in enumerate(boxes):
        x0, x1, y0, y1 = p.K
        wk = x1 - x0 + 1
        q = Q[m]
        for i, j in zip(*(v.tolist() for v in _ring(x0, x1, y0, y1))):
            at = (i - x0) + (j - y0) * wk
            hE, hN = (0.5 if j in by else 1.0), (0.5 if i in bx else 1.0)
            f = np.zeros(q.shape[1])
            if i < x1:
                f += aE[j, i] * hE * (q[at] - q[at + 1])
            if i > x0:
                f += aE[j, i - 1] * hE * (q[at] - q[at - 1])
            if j < y1:
                f += aN[j, i] * hN * (q[at] - q[at + wk])
            if j > y0:
                f += aN[j - 1, i] * hN * (q[at] - q[at - wk])
            held.setdefault((j, i), []).append((m, q[at], n * f))
    rows = sum(len(v) for v in held.values())
    P, d = np.zeros((rows, off[-1])), np.zeros((rows, phi.shape[0]))
    r = 0
    for (j, i), hs in held.items():
        if (i, j) in pos:
            for m, v, _ in hs:
                P[r, off[m]:off[m + 1]] = v
                d[r] = phi[:, pos[(i, j)]]
                r += 1
            continue
        for m, v, _ in hs[1:]:
            P[r, off[hs[0][0]]:off[hs[0][0] + 1]] = hs[0][1]
            P[r, off[m]:off[m + 1]] = -v
            r += 1
        for m, _, f in hs:
            P[r, off[m]:off[m + 1]] = f
        r += 1
    qq, rr = torch.linalg.qr(torch.from_numpy(P[:r]).cuda())
    c = torch.linalg.solve_triangular(rr, qq.T @ torch.from_numpy(d[:r]).cuda(), upper=True).cpu().numpy()
    u, cnt = np.zeros((phi.shape[0], n + 1, n + 1)), np.zeros((n + 1, n + 1))
    for m, p in enumerate(boxes):
        x0, x1, y0, y1 = p.K
        v = (Q[m] @ c[off[m]:off[m + 1]]).reshape(y1 - y0 + 1, x1 - x0 + 1, -1)
        u[:, y0:y1 + 1, x0:x1 + 1] += v.transpose(2, 0, 1)
        cnt[y0:y1 + 1, x0:x1 + 1] += 1
    u /= cnt
    u[:, rj, ri] = phi
    return u


def _exact_kinetic(case, seed):
    """Block elimination over the nodes, for the buffered patches at once and for the whole slab."""
    n, nv, M, W = case["n"], case["n_v"], case["patches"], case["n"] // case["patches"]
    v, w = np.polynomial.legendre.leggauss(nv)
    g, eps = case["g"], 2.0 ** -case["eps_log2"]
    k = 0.5 * (1 - g * g) / (1 + g * g + 2 * g * np.outer(v, v))
    A = np.diag(np.abs(v) * n + (w[:, None] * k).sum(0) / eps) - k * w[None, :] / eps
    up, dn = np.where(v > 0, v * n, 0.0), np.where(v < 0, -v * n, 0.0)

    def solve(cells, left, right):                       # left, right: (n_v, S) incoming values
        S = left.shape[1]
        Ws, ys = [], []
        for i in range(cells + 1):
            D, y = A.copy(), np.zeros((nv, S))
            L, U = up.copy(), dn.copy()
            if i == 0:
                D[v > 0] = np.eye(nv)[v > 0]
                y[v > 0] = left[v > 0]
            if i == cells:
                D[v < 0] = np.eye(nv)[v < 0]
                y[v < 0] = right[v < 0]
                U[:] = 0.0
            if i:
                D -= L[:, None] * Ws[-1]                  # Ws = Z^{-1} diag(U), ys = Z^{-1} y
                y += L[:, None] * ys[-1]
            s = np.linalg.solve(D, np.concatenate([np.diag(U), y], 1))
            Ws.append(s[:, :nv])
            ys.append(s[:, nv:])
        f = [ys[-1]]
        for i in range(cells - 1, -1, -1):
            f.append(ys[i] + Ws[i] @ f[-1])
        return np.stack(f[::-1])

    r = np.random.default_rng([seed, 3])
    inflow = 2.0 + r.standard_normal((1, 2, nv))
    full = solve(n, inflow[0, 0][:, None], inflow[0, 1][:, None])[..., 0]
    sigma = []
    for m in range(M):
        X0, X1 = max(0, m * W - case["buffer"]), min(n, (m + 1) * W + case["buffer"])
        z = _normals(seed, m, nv, case["samples"], 0x4D53504B)
        left, right = np.zeros_like(z), np.zeros_like(z)
        left[v > 0], right[v < 0] = z[:nv // 2], z[nv // 2:]
        R = solve(X1 - X0, left, right)[m * W - X0:m * W - X0 + W + 1].reshape(-1, case["samples"])
        sigma.append(np.linalg.svd(np.linalg.qr(R, mode="r"), compute_uv=False) if R.shape[0] >= R.shape[1]
                     else np.linalg.svd(R, compute_uv=False))
    return {"f": full[None], "sigma": np.concatenate(sigma), "k": None}


def exact(case, seed):
    if case["path"] == "kinetic":
        nodes = case["n"] + 2 * case["patches"] * case["buffer"]
        return _exact_kinetic(case, seed) if nodes * case["n_v"] ** 3 < 4e9 else None
    spec, boxes = _medium_spec(case, seed), _boxes(case)
    if case["path"] == "operator":
        aE, aN = _faces(case, spec)
        rows = max(p.X[3] - p.X[2] for p in boxes) + 1
        cols = max(p.X[1] - p.X[0] for p in boxes) + 1
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn((len(boxes), case["samples"], rows, (cols + 3) // 4 * 4), generator=g, device="cuda",
                        dtype=F64 if case["precision"] == "fp64" else torch.float32)
        y = torch.zeros(x.shape, dtype=F64, device="cuda")
        for m, p in enumerate(boxes):
            X0, X1, Y0, Y1 = p.X
            t = x[m, :, :Y1 - Y0 + 1, :X1 - X0 + 1].to(F64)
            c = t[:, 1:-1, 1:-1]
            y[m, :, 1:Y1 - Y0, 1:X1 - X0] = (
                aE[Y0 + 1:Y1, X0 + 1:X1] * (c - t[:, 1:-1, 2:]) + aE[Y0 + 1:Y1, X0:X1 - 1] * (c - t[:, 1:-1, :-2]) +
                aN[Y0 + 1:Y1, X0 + 1:X1] * (c - t[:, 2:, 1:-1]) + aN[Y0:Y1 - 1, X0 + 1:X1] * (c - t[:, :-2, 1:-1]))
        return y
    if case["path"] == "sample":
        if case["n"] > 1100:
            return None
        aE, aN = _faces(case, spec)
        return torch.cat([R.T.reshape(-1) for R in _snapshots(case, seed, boxes, aE, aN)])
    if case["n"] > 520 or 0.6 * sum(p.cols for p in boxes) > 7000:
        return None
    aE, aN = _faces(case, spec)
    Q, S = _bases(_snapshots(case, seed, boxes, aE, aN), case["tau"])
    u = _glue(case, boxes, aE, aN, Q, _phi(case, seed))
    return u if case["path"] in ("online", "map") else {"u": u, "sigma": np.concatenate(S), "k": None}
