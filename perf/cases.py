"""The work that users of the lgf library have it do, case by case.

A case is one pass of a program's own sequence of calls: links in, gauge
fixing, links out (``Lattice``), a batch of uneven lattices (``Batch``), links
from pinned host memory, overrelaxation sweeps, and one forward and backward
pass of the learned multiplier's network.  Handles, input links, output
buffers and weights are what such a program keeps between calls; ``prepare``
makes them.  Inputs are drawn from the recipe of the library's own workloads,
U_mu(x) = h(x) exp(i eps sum_a c_a lambda_a / 2) h^dag(x + mu^), with Haar h.

``exact`` repeats the calls with plain torch operations in complex128.
"""

import math

import numpy as np
import torch

from paper_1206_0675_gb300 import lgf, preconditioner

ALPHA = 0.08   # the step size of every workload of the library
OMEGA = 1.7    # overrelaxation parameter of its benchmark
OR_CHECK = 10  # sweeps between measurements of theta


def listed():
    fix = {"kind": "fix", "store12": False, "track": False, "learned": False, "tol": 0.0}
    return [
        # The smallest lattice of the library's configurations: one launch-bound fix.
        {**fix, "name": "fp64 8^4", "ext": "8x8x8x8", "prec": "fp64", "eps": 0.5, "n": 40, "track": True},
        # The headline lattice in plain FP64 with full matrices, an ordinary stretch of its loop.
        {**fix, "name": "fp64 32^4", "ext": "32x32x32x32", "prec": "fp64", "eps": 1.0, "n": 20},
        # Ragged extents (2s and 3s, none a warp wide), 12-real links, the transform tracked.
        {**fix, "name": "fp64-12 24x18x12x27 G", "ext": "24x18x12x27", "prec": "fp64", "eps": 0.8, "n": 20,
         "store12": True, "track": True},
        # The headline lattice in single precision, 12-real links: the phase that mixed runs spend most steps in.
        {**fix, "name": "fp32-12 32^4", "ext": "32x32x32x32", "prec": "fp32", "eps": 1.0, "n": 50, "store12": True},
        # The largest lattice of the library's configurations, single precision.
        {**fix, "name": "fp32-12 48^3x96", "ext": "48x48x48x96", "prec": "fp32", "eps": 0.7, "n": 10,
         "store12": True},
        # A whole fix to theta < 1e-15 in mixed precision, the transform tracked: what a user of smooth fields calls.
        {**fix, "name": "mixed 16^4 to 1e-15", "ext": "16x16x16x16", "prec": "mixed", "eps": 0.5, "n": 400,
         "store12": True, "track": True, "tol": 1e-15},
        # The learned multiplier with the shipped weights in FP64.
        {**fix, "name": "learned fp64 16^4", "ext": "16x16x16x16", "prec": "fp64", "eps": 0.7, "n": 20,
         "learned": True},
        # The other gauge-fixing method, FP64 and single precision.
        {"name": "or fp64 24^4", "kind": "or", "ext": "24x24x24x24", "prec": "fp64", "eps": 0.5, "n": 20,
         "store12": False},
        {"name": "or fp32-12 32^4", "kind": "or", "ext": "32x32x32x32", "prec": "fp32", "eps": 0.5, "n": 50,
         "store12": True},
        # Many small and middle lattices of uneven shapes in one call.
        {"name": "batch of 15", "kind": "batch", "ext": "8x8x8x8*6,12x12x12x12*4,16x16x16x16*4,16x16x16x32*1",
         "eps": 0.7, "n": 40},
        # One step at a time on links that arrive from pinned host memory.
        {"name": "host links fp64 32^4", "kind": "host", "ext": "32x32x32x32", "prec": "fp64", "eps": 1.0, "n": 1,
         "store12": False},
        # Forward and backward of the multiplier's network over a data set.
        {"name": "network loss and gradient", "kind": "grad", "n": 65536},
    ]


EXTENTS = [2, 3, 4, 6, 8, 9, 12, 16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 96]


def _draw_extents(rng, lo, hi, even=False):
    """Extents of factors 2 and 3 whose volume is spread over the logarithm of [lo, hi]."""
    allowed = [e for e in EXTENTS if e >= 4 and not (even and e % 2)]
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = target ** 0.25
    near = [e for e in allowed if side / 2.1 <= e <= side * 2.1]
    while True:
        ext = [rng.choice(near) for _ in range(4)]
        v = math.prod(ext)
        if target / 1.5 <= v <= min(hi, target * 1.5):
            return "x".join(map(str, ext)), v


def draw(rng):
    kind = rng.choice(["fix", "fix", "fix", "fix", "or", "batch", "host", "grad"])
    eps = round(rng.uniform(0.3, 1.0), 3)
    if kind == "grad":
        return {"kind": "grad", "n": int(math.exp(rng.uniform(math.log(4096), math.log(262144))))}
    if kind == "batch":
        shapes = []
        for _ in range(rng.randint(2, 4)):
            e, v = _draw_extents(rng, 2048, 131072)
            shapes.append("%s*%d" % (e, rng.randint(1, max(1, min(8, 131072 // v)))))
        return {"kind": "batch", "ext": ",".join(shapes), "eps": eps, "n": rng.randint(5, 40)}
    ext, v = _draw_extents(rng, 4096, 1 << 20, even=kind == "or")
    n = rng.randint(5, 50)
    prec = rng.choice(["fp64", "fp64", "fp32"])
    if prec == "fp64" and v > 200000:
        n = min(n, 20)  # no dearer than the largest listed case
    if prec == "fp32":  # theta stays well above the floor that single-precision links set it
        n, eps = min(n, 20), max(eps, 0.6)
    if kind == "host":
        return {"kind": "host", "ext": ext, "prec": prec, "eps": eps, "n": rng.randint(1, 3),
                "store12": rng.random() < 0.5}
    if kind == "or":
        return {"kind": "or", "ext": ext, "prec": prec, "eps": eps, "n": OR_CHECK * max(1, n // OR_CHECK),
                "store12": rng.random() < 0.5}
    return {"kind": "fix", "ext": ext, "prec": prec, "eps": eps, "n": n, "store12": rng.random() < 0.5,
            "track": rng.random() < 0.3, "learned": False, "tol": 0.0}


# --- inputs ------------------------------------------------------------------

def _ext(text):
    return tuple(int(e) for e in text.split("x"))


def _batch_exts(text):
    out = []
    for part in text.split(","):
        e, k = part.split("*")
        out += [_ext(e)] * int(k)
    return out


def _mm(a, b):
    out = a[..., :, 0:1] * b[..., 0:1, :]
    out += a[..., :, 1:2] * b[..., 1:2, :]
    out += a[..., :, 2:3] * b[..., 2:3, :]
    return out


def _dag(a):
    return a.conj().transpose(-1, -2)


def _rows_to_su3(r1, r2):
    """SU(3) matrix of two rows: Gram-Schmidt, third row (a x b)^*."""
    a = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    b = r2 - (a.conj() * r2).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b, dim=-1).conj()], dim=-2)


def _fwd(f, mu):
    return torch.roll(f, -1, dims=3 - mu)


def _back(f, mu):
    return torch.roll(f, 1, dims=3 - mu)


def _links(ext, eps, gen):
    lx, ly, lz, lt = ext
    dev = gen.device

    def gauss(*shape):
        return torch.complex(torch.randn(*shape, dtype=torch.float64, device=dev, generator=gen),
                             torch.randn(*shape, dtype=torch.float64, device=dev, generator=gen))

    z = gauss(lt, lz, ly, lx, 2, 3)
    h = _rows_to_su3(z[..., 0, :], z[..., 1, :])
    U = torch.empty((4, lt, lz, ly, lx, 3, 3), dtype=torch.complex128, device=dev)
    eye = torch.eye(3, dtype=torch.complex128, device=dev)
    s3 = math.sqrt(3.0)
    for mu in range(4):
        c = torch.randn(8, lt, lz, ly, lx, dtype=torch.float64, device=dev, generator=gen) * (0.5 * eps)
        X = torch.zeros((lt, lz, ly, lx, 3, 3), dtype=torch.complex128, device=dev)  # i H / 32
        X[..., 0, 0], X[..., 1, 1], X[..., 2, 2] = c[2] + c[7] / s3, -c[2] + c[7] / s3, -2 * c[7] / s3
        X[..., 0, 1], X[..., 0, 2], X[..., 1, 2] = (torch.complex(c[0], -c[1]), torch.complex(c[3], -c[4]),
                                                    torch.complex(c[5], -c[6]))
        for i, j in ((0, 1), (0, 2), (1, 2)):
            X[..., j, i] = X[..., i, j].conj()
        X *= 1j / 32.0
        E = eye + X / 10.0
        for k in range(9, 0, -1):
            E = eye + _mm(X, E) / k
        for _ in range(5):
            E = _mm(E, E)
        E = _mm(_mm(h, E), _dag(_fwd(h, mu)))
        U[mu] = _rows_to_su3(E[..., 0, :], E[..., 1, :])
    return U


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + 17)
    return g


def _network(n, seed):
    """Rows of the multiplier's data set: features, targets log m*, weights; He-initialised parameters."""
    gen = _generator(seed)
    X = torch.rand(n, 8, device="cuda", generator=gen)
    X[:, 6:] = 2 * X[:, 6:] - 1
    Y = torch.empty(n, device="cuda").uniform_(math.log(0.25), math.log(2.0), generator=gen)
    W = torch.rand(n, device="cuda", generator=gen) * 2
    P = torch.tensor(preconditioner.init_params(int(seed) % 100000), device="cuda")
    P[8896:8960] = torch.randn(64, device="cuda", generator=gen) * 0.1
    return P, X.contiguous(), Y, W


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grad":
        P, X, Y, W = _network(case["n"], seed)
        return {"case": case, "P": P, "X": X, "Y": Y, "W": W}
    gen = _generator(seed)
    if kind == "batch":
        exts = _batch_exts(case["ext"])
        U = [_links(e, case["eps"], gen) for e in exts]
        return {"case": case, "batch": lgf.Batch(exts), "U": U, "out": [torch.empty_like(u) for u in U]}
    ext = _ext(case["ext"])
    U = _links(ext, case["eps"], gen)
    lat = lgf.Lattice(ext, case["prec"], store12=case["store12"], track_G=bool(case.get("track")),
                      learned=bool(case.get("learned")))
    if case.get("learned"):
        lat.load_preconditioner(np.load(preconditioner.DEFAULT_WEIGHTS))
    state = {"case": case, "lat": lat, "out": torch.empty_like(U)}
    if case.get("track"):
        state["G"] = torch.empty(lat.site_shape, dtype=torch.complex128, device="cuda")
    state["U"] = U.cpu().pin_memory() if kind == "host" else U
    return state


# --- one pass ------------------------------------------------------------------

def _kept(case, t):
    """What a program keeps of a result: single precision where the handle computed in it (a mixed fix leaves a
    constant rotation of single-precision size, which the Landau gauge does not determine)."""
    return t if case["prec"] == "fp64" else t.to(torch.complex64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grad":
        grad = torch.empty(lgf.LGF_MLP_NPARAM, device="cuda")
        loss = lgf.lgf_mlp_loss_grad(state["P"].data_ptr(), state["X"].data_ptr(), state["Y"].data_ptr(),
                                     state["W"].data_ptr(), case["n"], grad.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        return {"loss": loss, "grad": grad}
    if kind == "batch":
        b = state["batch"]
        for i, U in enumerate(state["U"]):
            b.set_links(i, U)
        it, F, th, _ = b.fix(0.0, case["n"], ALPHA)
        for i, out in enumerate(state["out"]):  # the C interface: links into device memory
            st = lgf.load_library().lgf_batch_get_links(b.handle, i, out.data_ptr(), lgf.LGF_DEVICE)
            if st != lgf.LGF_OK:
                raise lgf.LgfError(st, "lgf_batch_get_links")
        return {"iters": it, "F": F, "theta": th, "links": state["out"]}
    lat = state["lat"]
    lat.set_links(state["U"])
    out = {}
    if kind == "host":
        for _ in range(case["n"]):
            lat.step(ALPHA)
        out["F"], out["theta"] = lat.measure()
    elif kind == "or":
        out["sweeps"], out["F"], out["theta"], _ = lat.or_fix(0.0, case["n"], OMEGA, OR_CHECK)
    else:
        out["iters"], out["F"], theta, _ = lat.fix(case["tol"], case["n"], ALPHA)
        if case["tol"] == 0.0:  # at a converged fix theta is rounding noise below tol
            out["theta"] = theta
    out["links"] = _kept(case, lat.get_links(state["out"]))
    if "G" in state:
        out["G"] = _kept(case, lat.get_transform(state["G"]))
    return out


# --- what a pass cannot do without ----------------------------------------------

def _site_work(ext, real_bytes, rows, kind):
    """Bytes and operations of one FA step or one overrelaxation sweep per site: links read and written once per
    step (once per colour for a sweep); for a step the packed divergence crosses memory for each of the two plane
    transforms there and back, with the update's two matrix products, the transforms, g and the measurement."""
    links = 4 * rows * 3 * 2 * real_bytes
    if kind == "or":
        return 2 * links, 4 * 2 * 198 + 600
    delta = 4 * 2 * real_bytes
    fft = 2 * 4 * 5 * math.log2(math.prod(ext))
    return 2 * links + 6 * delta, 4 * 2 * 198 + fft + 400


def work(case):
    if case["kind"] == "grad":
        n = case["n"]
        macs = 8 * 64 + 2 * 64 * 64 + 64
        return {"bytes": n * 10 * 4 + 2 * 8961 * 4, "flops": 6 * macs * n}
    exts = _batch_exts(case["ext"]) if case["kind"] == "batch" else [_ext(case["ext"])]
    prec = case.get("prec", "fp64")
    rb = 8 if prec == "fp64" else 4
    rows = 2 if case.get("store12") else 3
    n = case["n"]
    if case.get("tol"):
        n = 50  # about what a smooth field takes
    b = f = 0.0
    for e in exts:
        v = math.prod(e)
        sb, sf = _site_work(e, rb, rows, case["kind"])
        b += v * (n * sb + 2 * 576 + (144 if case.get("track") else 0))
        f += v * n * sf
    return {"bytes": b, "flops": f}


# --- the same calls in complex128 with plain torch --------------------------------

def _measure(U):
    """(divergence, F, theta) of links: D = sum_mu [A_mu(x - mu^) - A_mu(x)]."""
    V = U[0, ..., 0, 0].numel()
    W = torch.zeros_like(U[0])
    F = 0.0
    for mu in range(4):
        W += _back(U[mu], mu) - U[mu]
        F += float(torch.diagonal(U[mu], dim1=-2, dim2=-1).real.sum())
    D = (W - _dag(W)) / 2
    tr = torch.diagonal(D, dim1=-2, dim2=-1).sum(-1) / 3
    for i in range(3):
        D[..., i, i] -= tr
    return D, F / (12 * V), 4 * float(torch.view_as_real(D).square().sum()) / (3 * V)


def _filter(ext, dev):
    p2 = 0.0
    for mu, L in enumerate(ext):
        k = torch.arange(L, dtype=torch.float64, device=dev)
        shape = [1, 1, 1, 1]
        shape[3 - mu] = L
        p2 = p2 + (4 * torch.sin(math.pi * k / L) ** 2).reshape(shape)
    K = ALPHA * p2.max() / p2
    K[0, 0, 0, 0] = 0.0
    return K


def _gauge(U, g):
    return torch.stack([_mm(_mm(g, U[mu]), _dag(_fwd(g, mu))) for mu in range(4)])


def _exact_steps(U, ext, n, tol, track):
    K = _filter(ext, U.device)
    G = torch.eye(3, dtype=U.dtype, device=U.device).expand(U.shape[1:]).clone() if track else None
    D, F, th = _measure(U)
    it = 0
    while th >= tol and it < n:
        X = torch.empty_like(D)
        for i in range(2):
            for j in range(3):
                X[..., i, j] = torch.fft.ifftn(K * torch.fft.fftn(D[..., i, j]))
        X[..., 0, 0] += 1
        X[..., 1, 1] += 1
        g = _rows_to_su3(X[..., 0, :], X[..., 1, :])
        U = _gauge(U, g)
        if track:
            G = _mm(g, G)
        D, F, th = _measure(U)
        it += 1
    return U, G, it, F, th


def _exact_sweeps(U, ext, n):
    lx, ly, lz, lt = ext
    idx = [torch.arange(L, device=U.device) for L in (lt, lz, ly, lx)]
    par = (idx[0][:, None, None, None] + idx[1][:, None, None] + idx[2][:, None] + idx[3]) % 2
    eye = torch.eye(3, dtype=U.dtype, device=U.device)
    for _ in range(n):
        for parity in (0, 1):
            M = torch.zeros_like(U[0])
            for mu in range(4):
                M += U[mu] + _dag(_back(U[mu], mu))
            g = eye.expand(M.shape).clone()
            for i, j in ((0, 1), (0, 2), (1, 2)):
                b0 = M[..., i, i].real + M[..., j, j].real
                b1 = M[..., i, j].imag + M[..., j, i].imag
                b2 = M[..., i, j].real - M[..., j, i].real
                b3 = M[..., i, i].imag - M[..., j, j].imag
                r = torch.stack([b0, -b1, -b2, -b3])
                r = r / torch.linalg.vector_norm(r, dim=0)
                q = OMEGA * r
                q[0] += 1 - OMEGA
                q = q / torch.linalg.vector_norm(q, dim=0)
                a, b = torch.complex(q[0], q[3])[..., None], torch.complex(q[2], q[1])[..., None]
                for T in (M, g):
                    ti = a * T[..., i, :] + b * T[..., j, :]
                    tj = a.conj() * T[..., j, :] - b.conj() * T[..., i, :]
                    T[..., i, :], T[..., j, :] = ti, tj
            g = torch.where((par == parity)[..., None, None], g, eye)
            U = _gauge(U, g)
    _, F, th = _measure(U)
    return U, F, th


def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        P, X, Y, W = (t.double() for t in _network(case["n"], seed))
        P.requires_grad_(True)
        h = torch.relu(X @ P[0:512].reshape(64, 8).T + P[512:576])
        h = torch.relu(h @ P[576:4672].reshape(64, 64).T + P[4672:4736])
        h = torch.relu(h @ P[4736:8832].reshape(64, 64).T + P[8832:8896])
        z = h @ P[8896:8960] + P[8960]
        loss = (W * (torch.log(torch.nn.functional.softplus(z)) - Y) ** 2).sum() / case["n"]
        loss.backward()
        return {"loss": float(loss), "grad": P.grad}
    if case.get("learned"):
        return None  # the network runs in BF16 by design
    gen = _generator(seed)
    if kind == "batch":
        res = []
        for e in _batch_exts(case["ext"]):
            res.append(_exact_steps(_links(e, case["eps"], gen), e, case["n"], 0.0, False))
        return {"iters": None, "F": np.array([r[3] for r in res]), "theta": np.array([r[4] for r in res]),
                "links": [r[0] for r in res]}
    ext = _ext(case["ext"])
    U = _links(ext, case["eps"], gen)
    if kind == "or":
        U, F, th = _exact_sweeps(U, ext, case["n"])
        return {"sweeps": None, "F": F, "theta": th, "links": U}
    tol, n = case.get("tol", 0.0), case["n"]
    U, G, it, F, th = _exact_steps(U, ext, n, tol, bool(case.get("track")))
    out = {"F": F, "links": U}
    if tol == 0.0:
        out["theta"] = th
    if kind == "fix":
        out["iters"] = None
    if G is not None:
        out["G"] = G
    return out
