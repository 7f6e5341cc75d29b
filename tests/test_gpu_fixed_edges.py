"""Kernels at the ends of their range: values that are not finite, fields near
the identity, nearly dependent rows, long lines, long sums."""

import ctypes
import subprocess

import numpy as np
import pytest

from oracle import lgf_oracle as O
from paper_1206_0675_gb300 import build, fields, lgf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    lgf.load_library()


# Device functions that no entry point reaches by themselves, as a small library of their own.
PROBE = r"""
#include "lgf_or.cu"
using namespace lgf;
// G of one site after g with the given FP64 rows (stored as a lane stores them)
__global__ void accumulate(const double2* rows, double2* gf, double2* G) {
  fxg_store(gf, 1, 0, rows, rows + 3, rows + 6);
  accumulate_gauge_fx(1, 0, reinterpret_cast<const int4*>(gf), 1, G);
}
extern "C" int probe_accumulate(const double* rows, double* G) {
  double2* d;
  cudaMalloc(&d, 27 * sizeof(double2));
  cudaMemcpy(d, rows, 9 * sizeof(double2), cudaMemcpyHostToDevice);
  cudaMemcpy(d + 18, G, 9 * sizeof(double2), cudaMemcpyHostToDevice);
  accumulate<<<1, 1>>>(d, d + 9, d + 18);
  const cudaError_t e = cudaMemcpy(G, d + 18, 9 * sizeof(double2), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
// factors (i1, i2, kx, ky) of n sites from X = (f0, f1, f2, f3)
__global__ void factors(const float2* X, float4* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const GSFactorsOut o = gram_schmidt_pair(X[4 * i], X[4 * i + 1], X[4 * i + 2], X[4 * i + 3]);
  out[i] = make_float4(o.i1, o.i2, o.kx, o.ky);
}
extern "C" int probe_factors(const float* X, float* out, int n) {
  float2* d;
  cudaMalloc(&d, (size_t)n * 48);
  cudaMemcpy(d, X, (size_t)n * 32, cudaMemcpyHostToDevice);
  float4* o = reinterpret_cast<float4*>(d + (size_t)4 * n);
  factors<<<(n + 127) / 128, 128>>>(d, o, n);
  const cudaError_t e = cudaMemcpy(out, o, (size_t)n * 16, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
// a, b of the SU(2) hits on n blocks (of the local field over 16), and whether they are resolved
__global__ void hits(const double2* B, double2* out, int* ok, int n, double omega) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  FxC m[4], a, b;
  for (int k = 0; k < 4; ++k) m[k] = fx_from(B[4 * i + k]);
  const int64_t w7 = llrint(ldexp(7.0 * omega, 56)), c7 = llrint(ldexp(7.0 * (1.0 - omega), 56));
  bool good = true;
  or_subgroup_fx(m[0], m[1], m[2], m[3], fx_operand(w7), c7, a, b, good);
  out[2 * i] = make_double2(fx_value(a.x), fx_value(a.y));
  out[2 * i + 1] = make_double2(fx_value(b.x), fx_value(b.y));
  ok[i] = good;
}
extern "C" int probe_hits(const double* B, double* out, int* ok, int n, double omega) {
  double2* d;
  cudaMalloc(&d, (size_t)n * 7 * sizeof(double2));
  cudaMemcpy(d, B, (size_t)n * 64, cudaMemcpyHostToDevice);
  hits<<<(n + 127) / 128, 128>>>(d, d + 4 * n, reinterpret_cast<int*>(d + 6 * n), n, omega);
  cudaMemcpy(out, d + 4 * n, (size_t)n * 32, cudaMemcpyDeviceToHost);
  const cudaError_t e = cudaMemcpy(ok, d + 6 * n, (size_t)n * 4, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(PROBE)
    subprocess.run([build.nvcc(), "-shared", *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-o",
                    str(d / "libprobe.so"), str(d / "probe.cu")], check=True)
    return ctypes.CDLL(str(d / "libprobe.so"))


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


# ---------------------------------------------------------------------------
# a g that is not finite
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_transform_of_a_nonfinite_g(probe, bad):
    """G <- g G with an entry of g that is not finite is not finite, also where every sum that the entry's mark would
    enter as a number (-2) stays in range."""
    g = np.eye(3, dtype=np.complex128)
    g[1, 2] = bad
    G = np.full((3, 3), 0.3 + 0.2j)
    assert probe.probe_accumulate(ptr(g), ptr(G)) == 0
    assert not np.isfinite(G).any()


def test_transform_of_a_finite_g(probe):
    g = fields.random_links((2, 2, 2, 2), 0.9, seed=3).reshape(-1, 3, 3)[0]
    G = fields.random_links((2, 2, 2, 2), 0.9, seed=4).reshape(-1, 3, 3)[1].copy()
    want = g @ G
    assert probe.probe_accumulate(ptr(np.ascontiguousarray(g)), ptr(G)) == 0
    assert np.max(np.abs(G - want)) < 2e-15


# ---------------------------------------------------------------------------
# Gram-Schmidt factors of FP32 lanes on nearly dependent rows
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("A", [0.5, 4.0, 15.9, 16.1, 300.0, 4000.0])
def test_factors_of_nearly_dependent_rows(probe, A):
    """r1 = lambda r2 up to terms of order one, for entries up to A: i1 and i2 are the exact factors rounded once to
    FP32 (2^-24) after an error of 2^-35 (pairs) or 2^-53 |r2|^2 / |w|^2 < 2^-26 (FP64, entries up to 4000)."""
    n, rng = 20000, np.random.default_rng(5)
    z = lambda: rng.standard_normal(n) + 1j * rng.standard_normal(n)
    lam = rng.uniform(0.2, 1, n) * np.exp(2j * np.pi * rng.uniform(0, 1, n))
    lam[:n // 4] = np.exp(0.5j * np.pi * rng.integers(0, 4, n // 4))
    d = A * rng.uniform(0.5, 1, n) * rng.choice([-1, 1], n)
    f3 = A * rng.choice([0, 0.1, 0.7], n) * np.exp(2j * np.pi * rng.uniform(0, 1, n))
    f1 = 1j * lam * d + rng.choice([0, 0.3], n) * z()
    f2 = lam * f3 + rng.choice([0, 0.3], n) * z()
    X = np.stack([np.abs(lam) ** 2 * d, d, f1.real, f1.imag, f2.real, f2.imag, f3.real, f3.imag], axis=1)
    X = np.ascontiguousarray(np.clip(X, -A, A).astype(np.float32))
    out = np.empty((n, 4), dtype=np.float32)
    assert probe.probe_factors(ptr(X), ptr(out), n) == 0
    a, d, f1, f2, f3 = (x.astype(np.clongdouble) for x in
                        (X[:, 0], X[:, 1], X[:, 2] + 1j * X[:, 3].astype(np.clongdouble),
                         X[:, 4] + 1j * X[:, 5].astype(np.clongdouble), X[:, 6] + 1j * X[:, 7].astype(np.clongdouble)))
    r1, r2 = np.stack([1 + 1j * a, f1, f2]), np.stack([-np.conj(f1), 1 + 1j * d, f3])
    n1 = np.sum(np.abs(r1) ** 2, axis=0)
    w = r2 - np.sum(np.conj(r1) * r2, axis=0) / n1 * r1
    for got, want in ((out[:, 0], 1 / np.sqrt(n1)), (out[:, 1], 1 / np.sqrt(np.sum(np.abs(w) ** 2, axis=0)))):
        assert np.max(np.abs(got / want - 1)) < 1.25 * 2.0 ** -24


# ---------------------------------------------------------------------------
# gradient of the network over many chunks of samples
# ---------------------------------------------------------------------------

def test_network_gradient_of_many_equal_samples():
    """2^21 equal samples give the gradient of one.  Equal terms make every rounding of a sum push the same way: a
    sum of 64 samples, of up to 108 chunks, of 38 CTAs and of 8 parts is off by at most half of 2^-24 per term."""
    import torch
    n, rng = 1 << 21, np.random.default_rng(3)
    P = torch.from_numpy(np.ascontiguousarray(0.3 * rng.standard_normal(lgf.LGF_MLP_NPARAM), dtype=np.float32)).cuda()
    x = torch.from_numpy(rng.uniform(0.5, 1.5, (1, 8)).astype(np.float32)).cuda()
    grads = []
    for m in (1, n):
        X, Y, W = x.expand(m, 8).contiguous(), torch.full((m,), 0.7, device="cuda"), torch.ones(m, device="cuda")
        g = torch.empty(lgf.LGF_MLP_NPARAM, device="cuda")
        torch.cuda.synchronize()
        lgf.lgf_mlp_loss_grad(P.data_ptr(), X.data_ptr(), Y.data_ptr(), W.data_ptr(), m, g.data_ptr())
        grads.append(g.cpu().numpy().astype(np.float64))
    one, many = grads
    assert np.count_nonzero(one) > 1000
    assert np.all(np.abs(many - one) <= 0.5 * (64 + 108 + 38 + 8) * 2.0 ** -24 * np.abs(one))


# ---------------------------------------------------------------------------
# plans
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("ext, xc, threads", [((4, 2, 48, 96), 4, 768), ((2, 2, 128, 108), 2, 384),
                                              ((8, 12, 8, 6), 8, 64)])
def test_autotune_times_the_built_in_plan(ext, xc, threads):
    """The first trial is the plan an untuned handle runs: four x columns in one CTA that fills an SM, one tile
    between 220 and 227 KB, and an ordinary lattice."""
    with lgf.Lattice(ext, "fp32") as lat:
        lat.set_links(fields.random_links(ext, 0.8, seed=2))
        rep = lat.autotune()["fp32"]
    first = rep["candidates"][0]
    assert first["decomposition"] == "2d2d"
    assert (first["x_columns_zt"], first["threads"][1]) == (xc, threads)
    assert rep["candidates"][rep["chosen"]]["ms"] <= first["ms"]


# ---------------------------------------------------------------------------
# scratch of the network functions
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("make", [lambda: lgf.Lattice((4, 4, 4, 4), "fp64"), lambda: lgf.Batch([(4, 4, 4, 4)])])
def test_closing_a_handle_gives_back_the_network_scratch(make):
    import torch
    n, dev = 4096, "cuda"
    P, X = torch.zeros(lgf.LGF_MLP_NPARAM, device=dev), torch.ones(n, 8, device=dev)
    Y, W, g = torch.zeros(n, device=dev), torch.ones(n, device=dev), torch.empty(lgf.LGF_MLP_NPARAM, device=dev)
    torch.cuda.synchronize()
    args = [t.data_ptr() for t in (P, X, Y, W)] + [n, g.data_ptr()]
    lgf.lgf_mlp_loss_grad(*args)  # its code is loaded
    with lgf.Batch([(4, 4, 4, 4)]):
        pass
    lgf.Lattice((4, 4, 4, 4), "fp64").close()
    before = torch.cuda.mem_get_info()[0]
    lgf.lgf_mlp_loss_grad(*args)
    kept = before - torch.cuda.mem_get_info()[0]
    assert 0 < kept <= 64 << 20
    make().close()
    assert torch.cuda.mem_get_info()[0] == before


# ---------------------------------------------------------------------------
# lines of more than 64
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("ext, fp64", [((81, 81, 2, 2), 9.3e-16), ((72, 72, 2, 2), 8.0e-16), ((2, 2, 81, 81), 7.3e-16),
                                       ((2, 2, 128, 81), 9.6e-16), ((96, 72, 2, 2), 1.19e-15)])
def test_long_lines_are_no_further_off_than_fp64(ext, fp64):
    """g(x) of one step against extended precision: no further from it (rms, 5 % for another order of sums) than the
    same passes in FP64 arithmetic were on these links."""
    U = fields.random_links(ext, 0.9, seed=3)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    p2 = sum((4 * np.sin(pi * np.arange(L).astype(np.longdouble) / L) ** 2).reshape(
        [-1 if 3 - a == mu else 1 for a in range(4)]) for mu, L in enumerate(ext))
    K = np.longdouble(0.08) * p2.max() / np.where(p2 == 0, 1, p2)
    K[0, 0, 0, 0] = 0
    go = O.gauge_transform_from_divergence(O.divergence(U.astype(np.clongdouble)), K)
    with lgf.Lattice(ext, "fp64") as lat:
        lat.set_links(U)
        lat.step(0.08)
        g = lat.get_gauge()
    assert np.sqrt(np.mean(np.abs(g - go) ** 2)) < 1.05 * fp64


# ---------------------------------------------------------------------------
# hits of overrelaxation
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("omega", [1.0, 1.7, 1.999])
@pytest.mark.parametrize("size", [1.0, 0.3, 1e-3, 2.0 ** -20, 2.0 ** -21, 2.0 ** -22, 2.0 ** -40, 0.0])
def test_hits_down_to_where_their_direction_is_lost(probe, size, omega):
    """r^omega of blocks whose largest component is `size`: seven roundings of 2^-61 or less turn it, 2^-57 in all
    for the worst.  Below 2^-21 the site is handed to FP64."""
    n, rng = 2000, np.random.default_rng(8)
    v = rng.standard_normal((n, 4))
    v[:8] = np.concatenate([np.eye(4), -np.eye(4)])
    v = np.rint(v / np.max(np.abs(v), axis=1, keepdims=True) * size * 2.0 ** 59) * 2.0 ** -59
    B = np.zeros((n, 4), dtype=np.complex128)      # b0 .. b3 as sums of two entries each
    B[:, 0] = v[:, 0] / 2 + 1j * v[:, 3] / 2
    B[:, 3] = v[:, 0] / 2 - 1j * v[:, 3] / 2
    B[:, 1] = v[:, 2] / 2 + 1j * v[:, 1] / 2
    B[:, 2] = -v[:, 2] / 2 + 1j * v[:, 1] / 2
    out, ok = np.empty((n, 2), dtype=np.complex128), np.empty(n, dtype=np.int32)
    assert probe.probe_hits(ptr(B), ptr(out), ptr(ok), n, ctypes.c_double(omega)) == 0
    assert np.all(ok == (size >= 2.0 ** -21))
    if size < 2.0 ** -21:
        return
    r = np.stack([v[:, 0], -v[:, 1], -v[:, 2], -v[:, 3]], axis=1).astype(np.longdouble)
    r /= np.sqrt(np.sum(r * r, axis=1, keepdims=True))
    q = omega * r + np.array([1 - omega, 0, 0, 0])
    q /= np.sqrt(np.sum(q * q, axis=1, keepdims=True))
    got = np.stack([out[:, 0].real, out[:, 1].imag, out[:, 1].real, out[:, 0].imag], axis=1)
    assert np.max(np.abs(got - q)) < 2.0 ** -53 + 2.0 ** -57


@pytest.mark.parametrize("store12", [False, True])
@pytest.mark.parametrize("eps, fp64", [(0.25, 2.8e-32), (0.5, 1.15e-31)])
def test_or_converges_as_far_as_fp64(eps, fp64, store12):
    """theta of 8^4 levels off no higher than it did with hits in FP64 arithmetic (within 10 %)."""
    ext = (8, 8, 8, 8)
    with lgf.Lattice(ext, "fp64", store12=store12) as lat:
        lat.set_links(fields.random_links(ext, eps, seed=4))
        lat.or_sweep(1.7, 1500)
        theta = []
        for _ in range(15):
            lat.or_sweep(1.7, 1)
            theta.append(lat.measure()[1])
    assert np.median(theta) < 1.1 * fp64


# ---------------------------------------------------------------------------
# fields near the identity
# ---------------------------------------------------------------------------

def near(ext, eps, seed=4):
    return fields.random_links(ext, eps, seed=seed, gauge_rotate=False)


def floor_of_fix(ext, U, **kw):
    """theta after 250 steps, the median of the last 50."""
    decomposition = kw.pop("decomposition", None)
    with lgf.Lattice(ext, "fp64", **kw) as lat:
        if decomposition:
            lat.set_fft_decomposition(decomposition)
        lat.set_links(U)
        _, T = lat.set_trace(260)
        lat.fix(0.0, 250, 0.08)
    return np.median(T[200:250])


FORMS = [dict(), dict(store12=True), dict(exact_exp=True), dict(decomposition="1d4"), dict(track_G=True)]


@pytest.mark.parametrize("kw", FORMS, ids=lambda kw: "-".join(kw) or "plain")
@pytest.mark.parametrize("eps, fp64", [(1e-9, 3.9e-49), (1e-5, 3.8e-41), (1e-3, 3.9e-37), (0.03, 3.5e-34),
                                       (0.06, 1.4e-33), (0.12, 5.4e-33)])
def test_fix_near_the_identity_converges_as_far_as_fp64(eps, fp64, kw):
    """theta of 8^4 levels off no higher (10 %) than it does with every product and g in FP64 arithmetic."""
    ext = (8, 8, 8, 8)
    assert floor_of_fix(ext, near(ext, eps), **kw) < 1.1 * fp64


@pytest.mark.parametrize("store12", [False, True])
@pytest.mark.parametrize("eps, fp64", [(1e-9, 4.2e-49), (1e-5, 4.1e-41), (1e-3, 4.2e-37), (0.03, 3.9e-34),
                                       (0.06, 1.56e-33), (0.12, 6.3e-33)])
def test_or_near_the_identity_converges_as_far_as_fp64(eps, fp64, store12):
    ext = (8, 8, 8, 8)
    with lgf.Lattice(ext, "fp64", store12=store12) as lat:
        lat.set_links(near(ext, eps))
        lat.or_sweep(1.7, 1200)
        theta = []
        for _ in range(9):
            lat.or_sweep(1.7, 1)
            theta.append(lat.measure()[1])
    assert np.median(theta) < 1.1 * fp64


@pytest.mark.parametrize("ext", [(2, 2, 2, 2), (3, 4, 6, 9), (8, 8, 8, 8)])
@pytest.mark.parametrize("eps", [1e-9, 1e-4])
def test_gauge_near_the_identity_keeps_its_digits(eps, ext):
    """g - 1 of one step, of the size of eps, to the relative error of FP64 sums (1e-12 of its largest entry)."""
    U = near(ext, eps)
    D = O.divergence(U)
    go = O.gauge_transform_from_divergence(D, O.fa_filter(ext, 0.08))
    with lgf.Lattice(ext, "fp64") as lat:
        lat.set_links(U)
        lat.step(0.08)
        g = lat.get_gauge()
    off = ~np.eye(3, dtype=bool)
    assert np.max(np.abs(g - go)[..., off]) < 1e-12 * np.max(np.abs(go)[..., off])


PATCHES = {
    # warps of one kind, warps of both, single links
    "half": lambda x, y, z, t, mu: t < 1,
    "stripes": lambda x, y, z, t, mu: (x + y + z + t) % 2 == 0,
    "links": lambda x, y, z, t, mu: (x + 3 * y + 5 * z + 7 * t + mu) % 7 == 0,
}


@pytest.mark.parametrize("store12", [False, True])
@pytest.mark.parametrize("name", list(PATCHES))
@pytest.mark.parametrize("ext", [(2, 2, 2, 2), (6, 4, 2, 8), (8, 8, 6, 4), (32, 24, 6, 8)])
def test_fields_partly_near_the_identity(ext, name, store12):
    """Rough links with patches of links 1 + O(1e-6): measurement, step, transform and sweep against the oracle, with
    the bounds of the rough links (test_gpu_fixed.py)."""
    from oracle import lgf_or_oracle as R
    lx, ly, lz, lt = ext
    t, z, y, x = np.meshgrid(*(np.arange(n) for n in (lt, lz, ly, lx)), indexing="ij")
    U, W = fields.random_links(ext, 0.9, seed=3), near(ext, 1e-6)
    for mu in range(4):
        U[mu] = np.where(PATCHES[name](x, y, z, t, mu)[..., None, None], W[mu], U[mu])
    Us = U.copy()
    if store12:
        Us[..., 2, :] = np.conj(np.cross(U[..., 0, :], U[..., 1, :]))
    Fo, tho, Do = O.measure(Us)
    with lgf.Lattice(ext, "fp64", store12=store12, track_G=True) as lat:
        lat.set_links(U)
        F, th = lat.measure()
        D = lat.get_divergence()
        lat.step(0.08)
        g, U1, G1 = lat.get_gauge(), lat.get_links(), lat.get_transform()
        lat.set_links(U)
        lat.or_sweep(1.7, 1)
        U2, G2 = lat.get_links(), lat.get_transform()
    assert np.max(np.abs(D - Do)) < 4e-15 and abs(F - Fo) < 4e-15 and abs(th - tho) < 1e-13 * tho
    want = O.apply_gauge(Us, g)
    want[..., 2, :] = np.conj(np.cross(want[..., 0, :], want[..., 1, :]))
    assert np.max(np.abs(U1 - want)) < 2e-15
    assert np.max(np.abs(G1 - g)) < 2e-15
    Uo, Go = R.or_sweep(U, 1.7)
    assert np.max(np.abs(U2 - Uo)) < 1e-12 and np.max(np.abs(G2 - Go)) < 1e-12


def test_batch_and_mixed_near_the_identity():
    """A batch takes the steps of single handles to theta < 1e-38, and a mixed fix reaches it too."""
    exts = [(4, 4, 4, 4), (3, 4, 6, 9), (4, 4, 4, 4)]
    Us = [near(e, eps, seed=i) for i, (e, eps) in enumerate(zip(exts, (1e-5, 1e-5, 3e-6)))]
    with lgf.Batch(exts) as b:
        for i, U in enumerate(Us):
            b.set_links(i, U)
        it, F, th, conv = b.fix(1e-38, 400)
        links = [b.get_links(i) for i in range(3)]
    assert conv
    for i, (e, U) in enumerate(zip(exts, Us)):
        with lgf.Lattice(e, "fp64") as lat:
            lat.set_links(U)
            it1, F1, th1, conv1 = lat.fix(1e-38, 400, 0.08)
            assert conv1 and it1 == it[i] and np.array_equal(lat.get_links(), links[i])
        with lgf.Lattice(e, "mixed", store12=True) as lat:
            lat.set_links(U)
            assert lat.fix(1e-38, 400, 0.08)[3]
