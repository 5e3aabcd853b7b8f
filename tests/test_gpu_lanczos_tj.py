"""The Lanczos loop's FP64 scalars on the GPU: 1/x and x^{-1/2}, and
T_k^{1/2} e_1 with its stop test, each against long doubles (64 bits of
significand or more)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU test run without a CUDA device")
    from paper_1611_09322_gb300 import build
    so = str(tmp_path_factory.mktemp("tj") / "tj.so")
    subprocess.run([build.NVCC] + build.ARCH + ["-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I" + build.INCLUDE,
                    "-I" + build.CSRC, "-Xcompiler", "-fPIC", "-shared", os.path.join(HERE, "lanczos_tj.cu"), "-o", so,
                    "-lcudart"], check=True)
    return ctypes.CDLL(so)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _scalars(lib, x):
    r, q = np.empty_like(x), np.empty_like(x)
    assert lib.scalars_f64(len(x), _ptr(x), _ptr(r), _ptr(q)) == 0
    return r, q


def test_reciprocal_and_inverse_root(lib):
    """Random significands (and the ends of [1, 2)) at every exponent: 1/x to
    0.51 ulp and x^{-1/2} to 1.1 (its residual takes one rounded product more);
    zeros, denormals, infinities, NaN and negative roots as the operations."""
    rng = np.random.default_rng(1)
    m = np.concatenate([1.0 + rng.random(200), [1.0, 1.0 + EPS, 2.0 - EPS, 1.5, np.nextafter(4 / 3, 2)]])
    x = np.ldexp(m[None, :], np.arange(-1022, 1024)[:, None]).ravel()
    x = np.concatenate([x, -x])
    r, q = _scalars(lib, x)
    with np.errstate(invalid="ignore"):
        lx = x.astype(np.longdouble)
        rr, rq = 1 / lx, 1 / np.sqrt(lx)
    ok = np.abs(x) < 2.0 ** 1021  # 1/x is a normal number
    err = np.abs(r[ok].astype(np.longdouble) - rr[ok]) / np.spacing(np.abs(r[ok])).astype(np.longdouble)
    assert err.max() < 0.51, float(err.max())
    assert np.all(np.abs((r[~ok].astype(np.longdouble) - rr[~ok])) <= 5e-324)  # a denormal: to its last bit
    ok = x > 0
    err = np.abs(q[ok].astype(np.longdouble) - rq[ok]) / np.spacing(q[ok]).astype(np.longdouble)
    assert err.max() < 1.1, float(err.max())
    assert np.isnan(q[~ok]).all()
    s = np.array([0.0, -0.0, 5e-324, -5e-324, 1e-310, np.inf, -np.inf, np.nan])
    r, q = _scalars(lib, s)
    with np.errstate(all="ignore"):
        np.testing.assert_allclose(r, 1 / s, rtol=EPS)
        np.testing.assert_allclose(q, 1 / np.sqrt(s), rtol=2 * EPS)


def _sqrt_e1(al, be):
    """sqrt(T) e_1 = (2 / pi) int_0^inf T (T + t^2)^{-1} e_1 dt in long doubles,
    t = ||T||^{1/2} e^u: the trapezoidal rule converges like e^{-pi^2 / h}."""
    a, b = al.astype(np.longdouble), be.astype(np.longdouble)
    k, h = len(a), np.longdouble("0.2")
    t = np.sqrt(np.abs(a).max()) * np.exp(h * np.arange(-300, 301, dtype=np.longdouble))
    s, w = t * t, h * t * 2 / np.longdouble("3.14159265358979323846264338327950288")
    d = [None] * k
    d[k - 1] = a[k - 1] + s
    for i in range(k - 2, -1, -1):
        d[i] = a[i] + s - b[i] * b[i] / d[i + 1]
    x = 1 / d[0]
    y = [np.sum(w * (a[0] * x - (b[0] * b[0] * x / d[1] if k > 1 else 0)))]
    for i in range(1, k):
        x = -b[i - 1] * x / d[i]
        y.append(np.sum(-w * s * x))
    return np.array(y)


def _lanczos(lam, w):
    """The tridiagonal matrix with spectrum lam and weights w of e_1 (long
    double Lanczos on diag(lam), reorthogonalised)."""
    lam, q = lam.astype(np.longdouble), w.astype(np.longdouble) / np.sqrt(np.sum(w.astype(np.longdouble) ** 2))
    Q, al, be = [q], [], []
    for j in range(len(lam)):
        u = lam * Q[j]
        al.append(np.sum(u * Q[j]))
        for _ in range(2):
            for v in Q:
                u = u - np.sum(u * v) * v
        if j + 1 < len(lam):
            be.append(np.sqrt(np.sum(u * u)))
            Q.append(u / be[-1])
    return np.array(al, dtype=float), np.array(be, dtype=float)


def _run(lib, al, be, max_iter=64, fixed=64, tol=1e-3):
    K = len(al)
    y, ch, st = np.zeros((K, K)), np.zeros(K), np.zeros(K, dtype=np.int32)
    be = np.ascontiguousarray(be)
    assert lib.tj_sqrt_e1(K, _ptr(al), _ptr(be), max_iter, fixed, ctypes.c_double(tol), _ptr(y), _ptr(ch), _ptr(st)) == 0
    return y, ch, st


# spread of the spectrum: below 2^-18 of the scaled norm the QL route takes over
@pytest.mark.parametrize("spread", [3.0, 300.0, 2.0 ** 16, 2.0 ** 18 * 0.9, 2.0 ** 18 * 1.1, 2.0 ** 22])
@pytest.mark.parametrize("scale", [1.0, 0.0530516, 1e-9, 3e7])
def test_tj_sqrt_e1(lib, spread, scale):
    """Every k up to 64 (shared and global workspace, where they meet at 8 and
    9, and over- and underflowing determinants at the outer scales), on both
    sides of the hand-over to QL.  A backward error of eps ||T|| moves
    T^{1/2} e_1 by up to eps ||T|| / (2 lambda_min^{1/2}), against its norm
    alpha_1^{1/2} (e_1^T T e_1 is its square): the bound is eight of those
    (QL: j times as many rotations), and 8 eps.  The reported change and the
    stop rule are those of the returned vectors."""
    rng = np.random.default_rng(int(spread))
    for K in (1, 2, 5, 8, 9, 33, 64):
        lam = np.exp(rng.uniform(-np.log(spread), 0.0, K))
        lam[0] = 1.0
        if K > 1:
            lam[1] = 1.0 / spread
        al, be = _lanczos(lam * scale, rng.uniform(0.2, 1.0, K))
        y, ch, st = _run(lib, al, be)
        for k in sorted({1, 2, 3, 4, 7, 8, 9, 10, 32, 33, K}):
            if k > K:
                continue
            T = np.diag(al[:k]) + np.diag(be[:k - 1], 1) + np.diag(be[:k - 1], -1)
            ev = np.linalg.eigvalsh(T)
            ref = _sqrt_e1(al[:k], be[:k - 1])
            n = np.sqrt(np.sum(ref * ref))
            err = float(np.sqrt(np.sum((y[k - 1, :k] - ref) ** 2)) / n)
            bound = 8 * EPS * (1 + (1 + 0.25 * k) * ev[-1] / (2 * np.sqrt(ev[0])) / float(n))
            assert err < bound, (K, k, err, bound)
            if k > 1:
                d = y[k - 1, :k].copy()
                d[:k - 1] -= y[k - 2, :k - 1]
                assert ch[k - 1] == pytest.approx(np.linalg.norm(d) / np.linalg.norm(y[k - 1, :k]), rel=1e-12)
        tol = 0.5 * (ch[K // 2] + ch[K // 2 - 1]) if K > 4 else 1e-3
        st = _run(lib, al, be, max_iter=K, fixed=0, tol=tol)[2]
        want = [(k > 1 and ch[k - 1] < tol) or k >= K for k in range(1, K + 1)]
        assert list(st != 0) == want


@pytest.mark.parametrize("k", [3, 8, 9, 20])
def test_tj_zero_mode(lib, k):
    """A zero eigenvalue (coincident spheres) and one that rounding left
    slightly negative: square roots of max(lambda, 0); an eigenvalue's error of
    10 eps ||T|| moves its root by up to (10 eps)^{1/2}."""
    rng = np.random.default_rng(k)
    for low in (0.0, -1e-17):
        lam = np.concatenate([[low, 1.0], rng.uniform(0.1, 1.0, k - 2)])
        al, be = _lanczos(lam, rng.uniform(0.2, 1.0, k))
        y = _run(lib, al, be)[0][k - 1]
        l, Q = np.linalg.eigh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))
        ref = Q @ (np.sqrt(np.maximum(l, 0.0)) * Q[0])
        assert np.isfinite(y).all() and np.linalg.norm(y - ref) < 2 * np.sqrt(10 * EPS)
