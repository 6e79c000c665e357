"""The float64 grouped GEMM by digit products (csrc/gemm_digits.cuh): its
planner and its arithmetic on the CPU, the kernel on the GPU."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_20700_gb300", "csrc")


def test_planner(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path / "digit_plan_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, "-I", cuda_inc,
                    os.path.join(ROOT, "tests", "cpp", "digit_plan_check.cpp"),
                    os.path.join(CSRC, "gemm_digits_plan.cpp"), "-o", exe], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


# ------------------------------------------------------ the arithmetic, on CPU
def _digits(x):
    """Row exponents e (|x| < 2^e) and the eight balanced digits of
    F = round(x 2^(62-e)), rows x k, as the split kernel forms them."""
    big = np.abs(x).max(axis=1)
    e = np.where(big > 0, np.frexp(big)[1], 0)
    F = np.array([[int(v) for v in row] for row in np.floor(np.ldexp(np.abs(x).astype(np.longdouble), (62 - e)[:, None])
                                                            + np.longdouble(0.5))], dtype=object)
    F = np.where(x < 0, -F, F)
    d = np.zeros((8,) + x.shape, dtype=object)
    for s in range(7, 0, -1):
        d[s] = (F + 128) % 256 - 128
        F = (F - d[s]) // 256
    d[0] = F
    return e, d


def _graded(a, b):
    """The kernel's rule on op(A) and op(B)^T (rows x k both): operands graded
    along k go to the FMAs."""
    def expo(x):
        return np.where(x != 0, np.frexp(np.abs(x))[1], -10**6)
    ea, eb = expo(a), expo(b)
    ra, rb = ea - ea.max(axis=1)[:, None], eb - eb.max(axis=1)[:, None]
    ra[a == 0] = rb[b == 0] = -10**6
    rel, top = (ra.max(0) + rb.max(0)).max(), (ea.max(0) + eb.max(0)).max()
    return rel > -10**5 and (rel < -8 or top < ea.max() + eb.max() - 8)


def _product(a, b):
    """op(A) op(B) by the kernel's arithmetic; a: m x k, b: n x k."""
    ea, da = _digits(a)
    eb, db = _digits(b)
    h = np.zeros((a.shape[0], b.shape[0]), dtype=object)
    for k0 in range(0, a.shape[1], 256):
        for i in range(8):
            for j in range(8 - i):
                s = da[i][:, k0:k0 + 256] @ db[j][:, k0:k0 + 256].T
                h = h + s * 256 ** (7 - i - j)
        # what one FP32 accumulator holds stays an exact integer for d <= 4
        for d in range(5):
            acc = sum(np.abs(da[i][:, k0:k0 + 256]) @ np.abs(db[d - i][:, k0:k0 + 256]).T for i in range(d + 1))
            assert acc.max() <= 2**24
    v = np.array([[float(x) for x in row] for row in h])
    return np.ldexp(v, ea[:, None] + eb[None, :] - 68)


def _exact(a, b):
    fa = [[Fraction(float(x)) for x in r] for r in a]
    fb = [[Fraction(float(x)) for x in r] for r in b]
    return [[sum(x * y for x, y in zip(r, c)) for c in fb] for r in fa]


def _chain(a, b):
    c = np.zeros((a.shape[0], b.shape[0]))
    for k in range(a.shape[1]):
        c = c + a[:, k:k + 1] * b[:, k][None]
    return c


def _err(c, ex):
    """2-norm of c minus the rationals."""
    return float(np.linalg.norm([float(abs(Fraction(float(c[i, j])) - ex[i][j]))
                                 for i in range(c.shape[0]) for j in range(c.shape[1])]))


@pytest.mark.parametrize("k", [1, 7, 16, 17, 64, 257])
@pytest.mark.parametrize("kind", ["normal", "positive", "decay", "ints", "extreme digits", "rows scaled"])
def test_arithmetic_against_fma_chain(kind, k):
    """Digit products against exact rational sums: the error (2-norm) is at
    most that of a float64 multiply-add chain, or half an ulp per output."""
    rng = np.random.default_rng([k, len(kind)])
    m, n = 5, 4
    a, b = rng.standard_normal((m, k)), rng.standard_normal((n, k))
    if kind == "positive":
        a, b = np.abs(a), np.abs(b)
    elif kind == "decay":
        a *= np.exp(-np.abs(np.arange(k) * m / k - np.arange(m)[:, None]))
    elif kind == "ints":
        a, b = np.rint(9 * a), np.rint(9 * b)
    elif kind == "extreme digits":   # 0.498046875 = 0.0111...: digits of +-127, +-128
        a[:], b[:] = (2.0**53 - 1) / 2.0**53, -(1 - 2.0**-9 - 2.0**-17 - 2.0**-25 - 2.0**-33)
    elif kind == "rows scaled":
        a *= 10.0 ** np.linspace(-60, 60, m)[:, None]
    ex = _exact(a, b)
    if _graded(a, b):
        assert kind == "decay"
        return
    c = _product(a, b)
    half_ulp = float(np.linalg.norm([float(abs(x)) * 2.0**-53 for r in ex for x in r]))
    assert _err(c, ex) <= max(_err(_chain(a, b), ex), 1.01 * half_ulp)


def test_graded_operands_are_found():
    rng = np.random.default_rng(2)
    a, b = rng.standard_normal((6, 40)), rng.standard_normal((7, 40))
    g = 10.0 ** np.linspace(-60, 60, 40)
    assert not _graded(a, b)
    assert _graded(a * g, b / g)
    assert not _graded(a * 10.0 ** np.linspace(-90, 90, 6)[:, None], b)
    a[:, 20:], b[:, :20] = 0.0, 0.0   # no common column: an exact zero either way
    assert not _graded(a, b)


# ---------------------------------------------------------------- on the GPU
@pytest.fixture(scope="module")
def pkg():
    import paper_2503_20700_gb300 as p
    p.load()
    return p


def _run(pkg, a, b, ta, tb, alpha=1.0, pad=0, C0=None):
    """a: m x k, b: k x n, stored either way round with `pad` extra columns."""
    def stored(x, t):
        x = x.T if t else x
        s = np.full((x.shape[0], x.shape[1] + pad), np.nan)
        s[:, :x.shape[1]] = x
        return s
    A, B = stored(a, ta), stored(b, tb)
    m, k, n = a.shape[0], a.shape[1], b.shape[1]
    C = np.zeros((m, n + pad)) if C0 is None else C0.copy()
    pkg.ops.grouped_gemm(A.ravel(), B.ravel(), C, [(0, m, n, C.shape[1], 0, 1)],
                         [(0, 0, k, A.shape[1], B.shape[1], ta, tb, alpha)])
    return C


@pytest.mark.gpu
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("m,n,k", [(128, 64, 256), (127, 65, 255), (129, 63, 257), (200, 16, 512), (257, 130, 33),
                                   (70, 200, 513), (96, 97, 1000), (64, 48, 64)])
def test_kernel_against_longdouble(pkg, m, n, k, ta, tb):
    """Edges of tiles, chunks (256 terms) and 16-column steps, padded leading
    dimensions, C added to.  Each output is rounded once from the exact sum of
    the digits and once by the addition to C: 2^-53 of each."""
    rng = np.random.default_rng([m, n, k, ta, tb])
    a, b = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    C0 = rng.standard_normal((m, n + 3))
    C = _run(pkg, a, b, ta, tb, alpha=-0.75, pad=3, C0=C0)
    assert np.array_equal(C[:, n:], C0[:, n:])
    rows = rng.choice(m, min(m, 8), replace=False)
    ref = -0.75 * (a[rows].astype(np.longdouble) @ b.astype(np.longdouble))
    err = np.abs(C[rows, :n] - (C0[rows, :n] + ref)).astype(float)
    # sqrt(k) 2^-62 of the row maxima's product for what the split drops
    drop = np.sqrt(k) * 2.0**-60 * np.abs(a).max() * np.abs(b).max()
    assert np.all(err <= 2.0**-53 * (np.abs(ref) + np.abs(C0[rows, :n] + ref)).astype(float) + drop)


@pytest.mark.gpu
def test_kernel_many_segments(pkg):
    """Few tiles and many segments (partial tiles, reduced in order): equal to
    numpy, bitwise reproducible."""
    rng = np.random.default_rng(4)
    S, m, n, k = 61, 150, 70, 90
    A, B = rng.standard_normal((S, m, k)), rng.standard_normal((S, k, n))
    C0 = rng.standard_normal((m, n))
    segs = [(i * m * k, i * k * n, k, k, n, 0, 0, 0.5) for i in range(S)]
    C1, C2 = C0.copy(), C0.copy()
    for C in (C1, C2):
        pkg.ops.grouped_gemm(A.ravel(), B.ravel(), C, [(0, m, n, n, 0, S)], segs)
    ref = C0 + 0.5 * np.einsum("sik,skj->ij", A, B)
    assert np.array_equal(C1, C2)
    assert np.abs(C1 - ref).max() <= 2 * np.sqrt(S * k) * 2.0**-53 * np.sqrt(S * k) * 4
    one = C0.copy()
    pkg.ops.grouped_gemm(A.ravel(), B.ravel(), one, [(0, m, n, n, 0, 0)], segs)
    assert np.array_equal(one, C0)


@pytest.mark.gpu
def test_kernel_special_operands(pkg):
    """Non-finite entries, operands graded along k, extreme row scales and
    zero rows: the float64 FMAs' answers."""
    rng = np.random.default_rng(6)
    m, n, k = 130, 80, 300
    a, b = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    x = a.copy()
    x[3, 5], x[7, 9], x[11, 2] = np.inf, np.nan, -np.inf
    with np.errstate(invalid="ignore"):
        ref = x @ b
    C = _run(pkg, x, b, 0, 0)
    assert np.array_equal(np.isnan(C), np.isnan(ref))
    ok = ~np.isnan(ref)
    assert np.array_equal(np.isinf(C[ok]), np.isinf(ref[ok])) and np.array_equal(np.sign(C[3]), np.sign(ref[3]))
    fin = np.isfinite(ref)
    assert np.abs(C[fin] - ref[fin]).max() <= k * 2.0**-53 * (np.abs(a) @ np.abs(b)).max()
    g = 10.0 ** np.linspace(-60, 60, k)
    for y, z in [(a * g, b / g[:, None]), (a * 1e200, b), (a * 1e-250, b * 1e200),
                 (a * 10.0 ** np.linspace(-90, 90, m)[:, None], b)]:
        C = _run(pkg, y, z, 1, 0)
        scale = np.abs(y) @ np.abs(z)
        assert np.all(np.abs(C - y @ z) <= 2 * k * 2.0**-53 * scale)
    y = a.copy()
    y[5], y[:, 7] = 0.0, 0.0
    C = _run(pkg, y, b, 0, 1)
    assert np.all(C[5] == 0.0) and np.abs(C - y @ b).max() <= 2 * k * 2.0**-53 * (np.abs(y) @ np.abs(b)).max()
    assert np.all(_run(pkg, np.zeros((m, k)), b, 0, 0) == 0.0)
