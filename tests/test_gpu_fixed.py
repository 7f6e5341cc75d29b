"""The fixed-point forms of the FP64 kernels against the FP64 oracle, where
they can go wrong: entries of exactly 0, 1, -1 and i, entries far below the
fixed-point unit, lattices that do not fill a CTA, and values outside the
fixed-point range (an infinite step), which take the FP64 path.

Tolerances: a link of the update is two sums of three complex products and
one FP64 rounding of entries of order one, 2^-53 + a few 2^-58 against the
oracle's own 2^-53 per operation: 2e-15 covers both.  A divergence entry adds
16 link entries: 4e-15.
"""

import numpy as np
import pytest

from oracle import lgf_oracle as O
from paper_1206_0675_gb300 import fields, lgf

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    lgf.load_library()


def permutation_links(ext, seed):
    """Links with one entry of 1, -1, i or -i per row and column, determinant 1."""
    rng = np.random.default_rng(seed)
    lx, ly, lz, lt = ext
    shape = (4, lt, lz, ly, lx)
    U = np.zeros(shape + (3, 3), dtype=np.complex128)
    perms = np.array([(0, 1, 2), (1, 2, 0), (2, 0, 1), (0, 2, 1), (1, 0, 2), (2, 1, 0)])
    p = perms[rng.integers(0, 6, shape)]
    ph = rng.integers(0, 4, shape + (3,))
    odd = np.isin(np.arange(6), (3, 4, 5))[(p[..., None, :] == perms).all(-1).argmax(-1)]
    ph[..., 2] = (-ph[..., 0] - ph[..., 1] + 2 * odd) % 4
    vals = np.array([1, 1j, -1, -1j])[ph]
    for r in range(3):
        np.put_along_axis(U[..., r, :], p[..., r:r + 1], vals[..., r:r + 1], axis=-1)
    return U


def rebuilt(U):
    """Row 3 from rows 1-2, (a x b)^*: what 12-real storage holds, and the row 3 of every updated link."""
    V = U.copy()
    V[..., 2, :] = np.conj(np.cross(U[..., 0, :], U[..., 1, :]))
    return V


def weak_links(ext, eps):
    return fields.random_links(ext, eps, seed=4, gauge_rotate=False)


CASES = {
    "permutations": lambda ext: permutation_links(ext, 1),
    "weak 1e-3": lambda ext: weak_links(ext, 1e-3),
    "weak 1e-9": lambda ext: weak_links(ext, 1e-9),
    "weak 1e-19": lambda ext: weak_links(ext, 1e-19),
    "random": lambda ext: fields.random_links(ext, 0.9, seed=3),
}


@pytest.mark.parametrize("store12", [False, True])
@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("ext", [(2, 2, 2, 2), (3, 4, 6, 9), (8, 8, 4, 2)])
def test_measure_and_step_against_oracle(ext, name, store12):
    U = CASES[name](ext)
    Us = rebuilt(U) if store12 else U
    Fo, tho, Do = O.measure(Us)
    with lgf.Lattice(ext, "fp64", store12=store12) as lat:
        lat.set_links(U)
        F, th = lat.measure()
        D = lat.get_divergence()
        lat.step(0.08)
        g = lat.get_gauge()
        U1 = lat.get_links()
    assert np.max(np.abs(D - Do)) < 4e-15
    assert abs(F - Fo) < 4e-15
    assert abs(th - tho) < 1e-13 * tho
    assert np.max(np.abs(U1 - rebuilt(O.apply_gauge(Us, g)))) < 2e-15


@pytest.mark.parametrize("store12", [False, True])
def test_infinite_step_is_reported(store12):
    ext = (4, 4, 4, 4)
    with lgf.Lattice(ext, "fp64", store12=store12) as lat:
        lat.set_links(fields.random_links(ext, 0.9, seed=3))
        lat.step(1e308)
        with pytest.raises(lgf.LgfError) as e:
            lat.measure()
        assert e.value.status == lgf.LGF_E_NONFINITE


# ---------------------------------------------------------------------------
# plane passes in block floating point
# ---------------------------------------------------------------------------

def fields4(ext, seed=7):
    lx, ly, lz, lt = ext
    rng = np.random.default_rng(seed)
    shape = (4, lt, lz, ly, lx)
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def fft_ref(f, sign):
    axes = (1, 2, 3, 4)
    return np.fft.fftn(f, axes=axes) if sign < 0 else np.fft.ifftn(f, axes=axes, norm="forward")


INPUTS = {
    "random": lambda f: f,
    "constant": lambda f: 1.0 + 1e-3 * f,
    "one site": lambda f: np.where(np.arange(f[0].size).reshape(f[0].shape) == f[0].size - 1, f, 0.0),
    # planes of very different size: every (x,y) plane and every (z,t) plane has its own exponent
    "wide range": lambda f: f * 10.0 ** (8 * np.sin(np.arange(f[0].size).reshape(f[0].shape))),
    # the ends of the FP64 range
    "1e-300": lambda f: 1e-300 * f,
    "1e300": lambda f: 1e300 * f,
    "zero": lambda f: 0.0 * f,
}


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("name", list(INPUTS))
@pytest.mark.parametrize("ext", [(2, 2, 2, 2), (3, 4, 6, 9), (8, 27, 2, 16), (32, 4, 24, 3), (81, 2, 3, 64)])
def test_fft4_block_floating_point(ext, name, sign):
    """Norm-wise error below 1e-15: FP64's own (numpy's) is up to 5e-16, ours below 3e-16."""
    f = np.ascontiguousarray(INPUTS[name](fields4(ext)))
    scale = np.max(np.abs(f)) or 1.0
    ref = fft_ref(f / scale, sign)
    with lgf.Lattice(ext, "fp64") as lat:
        got = lat.fft4(f, sign) / scale
    if name == "zero":
        assert not np.any(got)
        return
    assert np.linalg.norm(got - ref) < 1e-15 * np.linalg.norm(ref)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_fft4_nonfinite_input(bad):
    """One bad site spoils its own field and no other."""
    ext = (4, 6, 3, 8)
    f = fields4(ext)
    f[2, 1, 0, 2, 3] = bad
    with lgf.Lattice(ext, "fp64") as lat:
        got = lat.fft4(f, -1)
    assert not np.any(np.isfinite(got[2]))
    ref = fft_ref(f[[0, 1, 3]], -1)
    assert np.linalg.norm(got[[0, 1, 3]] - ref) < 1e-15 * np.linalg.norm(ref)


# ---------------------------------------------------------------------------
# overrelaxation
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("omega", [1.0, 1.7, 1.999])
@pytest.mark.parametrize("name", ["random", "weak 1e-3", "weak 1e-9"])
@pytest.mark.parametrize("ext", [(2, 2, 2, 2), (2, 2, 4, 6), (4, 6, 2, 8)])
def test_or_sweep_against_oracle(ext, name, omega):
    """One sweep (both colours), with and without row 3 and the transform, at site counts that end inside a CTA;
    links within the rounding of the two sides, 1e-12 as for the other sweeps."""
    from oracle import lgf_or_oracle as R
    U = CASES[name](ext)
    Uo, Go = R.or_sweep(U, omega)
    for store12 in (False, True):
        with lgf.Lattice(ext, "fp64", store12=store12, track_G=True) as lat:
            lat.set_links(U)
            lat.or_sweep(omega, 1)
            U1, G = lat.get_links(), lat.get_transform()
        assert np.max(np.abs(U1 - Uo)) < 1e-12
        assert np.max(np.abs(G - Go)) < 1e-12


# ---------------------------------------------------------------------------
# links in and out
# ---------------------------------------------------------------------------

@pytest.mark.parametrize("where", [0, 1, 130, 2591])
@pytest.mark.parametrize("bad", [False, True])
def test_su3_check_accepts_and_rejects_by_its_bound(where, bad):
    """|det U - 1| = 3 eps of one scaled matrix just below and just above 1e-10, first, last and inside a tile."""
    ext = (3, 4, 6, 9)
    U = fields.random_links(ext, 0.8, seed=6)
    U.reshape(-1, 3, 3)[where] *= 1 + (3.4e-11 if bad else 3.25e-11)
    with lgf.Lattice(ext, "fp64") as lat:
        if bad:
            with pytest.raises(lgf.LgfError) as e:
                lat.set_links(U)
            assert e.value.status == lgf.LGF_E_ARG
        else:
            lat.set_links(U)


@pytest.mark.parametrize("name", ["random", "permutations", "weak 1e-40"])
@pytest.mark.parametrize("ext", [(2, 2, 2, 2), (3, 4, 6, 9)])
def test_links_round_trip(ext, name):
    """FP64 links come back as they went in, FP32 links as their IEEE rounding (zeros and subnormals among them)."""
    U = weak_links(ext, 1e-40) if name == "weak 1e-40" else CASES[name](ext)
    with lgf.Lattice(ext, "fp64") as lat:
        lat.set_links(U)
        assert np.array_equal(lat.get_links(), U)
    with lgf.Lattice(ext, "fp32") as lat:
        lat.set_links(U)
        assert np.array_equal(lat.get_links(), U.astype(np.complex64).astype(np.complex128))


# ---------------------------------------------------------------------------
# Gram-Schmidt of FP32 lanes in FP32 pairs
# ---------------------------------------------------------------------------

def check_fp32_gauge(ext, alpha):
    """g(x) of one FP32 step against the oracle.

    Tolerance: the filtered field is known to about 1e-6 of its size (FP32
    divergence and transforms), which row 2 minus its projection on row 1
    amplifies by |r2| / |w|; 5e-6 of that covers the rounding of g as well.
    """
    U = fields.random_links(ext, 0.9, seed=3)
    D, K = O.divergence(U), O.fa_filter(ext, alpha)
    go = O.gauge_transform_from_divergence(D, K)
    M = O.ifft4(O.fft4(D) * K[..., None, None]) + np.eye(3)
    r2 = M[..., 1, :]
    ip = np.sum(np.conj(go[..., 0, :]) * r2, axis=-1)
    kappa = np.linalg.norm(r2, axis=-1) / np.linalg.norm(r2 - ip[..., None] * go[..., 0, :], axis=-1)
    with lgf.Lattice(ext, "fp32") as lat:
        lat.set_links(U)
        lat.step(alpha)
        g = lat.get_gauge()
    assert np.all(np.abs(g - go).max(axis=(-1, -2)) < 5e-6 * kappa)


@pytest.mark.parametrize("alpha", [1e-6, 0.08, 3.0, 3e3, 3e7])
def test_fp32_gauge_against_oracle(alpha):
    """alpha = 3e3 puts sites on both sides of the pairs' range, 3e7 all beyond it."""
    check_fp32_gauge((3, 4, 6, 9), alpha)


# ---------------------------------------------------------------------------
# plane passes of FP32 lanes on pairs
# ---------------------------------------------------------------------------

PAIR_EXTS = [(2, 2, 2, 2), (3, 27, 2, 4), (6, 3, 12, 9), (8, 12, 6, 16), (16, 18, 4, 8), (36, 4, 2, 48),
             (54, 2, 24, 3), (2, 96, 64, 2), (4, 2, 72, 108), (4, 2, 48, 96)]


@pytest.mark.parametrize("ext", PAIR_EXTS)
def test_fp32_plane_passes_against_oracle(ext):
    """Every radix, one and several stages a line, odd extents, one column pair and several."""
    check_fp32_gauge(ext, 0.08)


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("ext", PAIR_EXTS)
def test_fp32_transform_against_reference(ext, sign):
    """FP32 transforms in natural order: rounding grows with the stages, 2^-24 each of at most 16."""
    f = fields4(ext)
    ref = fft_ref(f, sign)
    with lgf.Lattice(ext, "fp32") as lat:
        out = lat.fft4(f, sign)
    assert np.linalg.norm(out - ref) < 16 * 2 ** -24 * np.linalg.norm(ref)


@pytest.mark.parametrize("ext", [(81, 81, 2, 2), (2, 2, 81, 54), (64, 64, 2, 2)])
def test_fp64_gauge_of_long_lines(ext):
    """g(x) of one FP64 step against extended precision, where the filter weights the lowest modes most.

    A rounding that is not centred adds up in those modes.  A plane of N elements
    in units of 2^-53 of its largest gathers sqrt(N) rounding errors of 0.3 units:
    2.7e-15 for 81 x 81 and a filtered field of order one; 4e-15 in the 2-norm.
    """
    U = fields.random_links(ext, 0.9, seed=3)
    Ux = U.astype(np.clongdouble)
    p2 = sum((4 * np.sin(np.pi * np.arange(L).astype(np.longdouble) / L) ** 2).reshape(
        [-1 if 3 - a == mu else 1 for a in range(4)]) for mu, L in enumerate(ext))
    K = np.longdouble(0.08) * p2.max() / np.where(p2 == 0, 1, p2)
    K[0, 0, 0, 0] = 0
    go = O.gauge_transform_from_divergence(O.divergence(Ux), K)
    with lgf.Lattice(ext, "fp64") as lat:
        lat.set_links(U)
        lat.step(0.08)
        g = lat.get_gauge()
    assert np.sqrt(np.mean(np.abs(g - go) ** 2)) < 4e-15
