"""The error weights of the step-size control: their device functions against
correctly rounded division and an extended-precision power, and solves with
atol = 0 whose smallest entries have weights below the range of a reciprocal.

Bounds.  ratio, FP64: the cubic step leaves less than 2^-60 of an approximation
good to 2^-20, so the reciprocal carries its last rounding and the product one
more: at most 2 ulp from the rounded quotient (subnormal quotients: 2 units of
2^-1074).  FP32: rcp.approx is within an ulp and the product rounds once, so
2^-22 relative (subnormal: 2 units of 2^-149).  inv_root10: the seed is good to
1e-6, which leaves 4e-17; the rounding of x y^10 (5 operations of 2^-53) counts
a tenth and the last operation half an ulp: 4e-16 relative over [1.6e-8, 1e7],
the squared errors that the step control passes to it."""
import os
import subprocess

import numpy as np
import pytest

from paper_1110_0573_gb300 import systems as S

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def qt():
    from paper_1110_0573_gb300 import build
    build.build()
    from paper_1110_0573_gb300 import qt as q
    return q


@pytest.fixture(scope="module")
def device_math(qt, tmp_path_factory):
    from paper_1110_0573_gb300 import build
    tmp = tmp_path_factory.mktemp("devmath")
    exe = str(tmp / "device_math_check")
    r = subprocess.run([build.nvcc(), "-std=c++17", "-O3", *build.ARCH,
                        os.path.join(ROOT, "tests", "device_math_check.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]

    def run(x, w, r10):
        src, dst = str(tmp / "in"), str(tmp / "out")
        with open(src, "wb") as f:
            np.array([len(x)], dtype=np.int64).tofile(f)
            for a in (x, w, r10):
                np.ascontiguousarray(a, dtype=np.float64).tofile(f)
        assert subprocess.run([exe, src, dst]).returncode == 0
        return np.fromfile(dst, dtype=np.float64).reshape(3, -1)

    return run


def exponents(rng, n, edges, lo, hi):
    """n positive numbers 2^e m, e over [lo, hi] and around the edges."""
    e = np.concatenate([rng.uniform(lo, hi, n // 2), rng.choice(edges, n - n // 2) +
                        rng.choice([-2, -1, 0, 1, 2], n - n // 2)])
    return np.ldexp(rng.uniform(1.0, 2.0, n), np.clip(e, lo, hi).astype(int))


def test_ratio_fp64(device_math):
    rng = np.random.default_rng(1)
    n = 400_000
    w = exponents(rng, n, [-1007, 993, -1022, 1022, 0], -1073, 1022)
    w[:6] = [0.0, np.inf, np.nan, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308]
    with np.errstate(over="ignore"):
        x = w * rng.uniform(-4.0, 4.0, n)  # quotients of order one, as the controller forms them
    x[n // 2:] = exponents(rng, n - n // 2, [0], -1073, 1022)  # and any
    x[:6] = [1.0, 1.0, 1.0, 1e-323, 1.0, -1.7976931348623157e308]
    got = device_math(x, w, np.ones(n))[0]
    with np.errstate(all="ignore"):
        want = x / w
    special = ~np.isfinite(want)
    assert np.array_equal(got[special], want[special], equal_nan=True)
    err = np.abs(got[~special] - want[~special])
    assert (err <= 2 * np.spacing(np.abs(want[~special]))).all()


def test_ratio_fp32(device_math):
    rng = np.random.default_rng(2)
    n = 400_000
    w = exponents(rng, n, [-126, 126, 0], -148, 126).astype(np.float32)
    w[:5] = [0.0, np.inf, np.nan, 1e-45, 1.1754944e-38]
    with np.errstate(over="ignore"):
        x = (w * rng.uniform(-4.0, 4.0, n)).astype(np.float32)
    x[n // 2:] = exponents(rng, n - n // 2, [0], -148, 126).astype(np.float32)
    x[:5] = [1.0, 1.0, 1.0, 3e-45, 1.0]
    got = device_math(x, w, np.ones(n))[1].astype(np.float32)
    with np.errstate(all="ignore"):
        want = x / w
    special = ~np.isfinite(want) | ~np.isfinite(got)
    with np.errstate(all="ignore"):  # within the bound of the largest number: either
        top = np.abs(x.astype(np.float64) / w) >= np.finfo(np.float32).max * (1 - 2.0 ** -22)
    assert np.array_equal(got[special & ~top], want[special & ~top], equal_nan=True)
    ok = ~special
    err = np.abs(got[ok].astype(np.float64) - want[ok])
    assert (err <= np.maximum(2.0 ** -22 * np.abs(want[ok].astype(np.float64)), 2 * 2.0 ** -149)).all()


def test_inv_root10(device_math):
    rng = np.random.default_rng(3)
    n = 400_000
    x = np.exp(rng.uniform(np.log(1.6e-8), np.log(1e7), n))
    x[:3] = [1.6e-8, 1.0, 1e7]
    got = device_math(np.ones(n), np.ones(n), x)[2]
    want = np.power(x.astype(np.longdouble), np.longdouble(-1) / 10)
    assert (np.abs(got - want) <= 4e-16 * want).all()


H = np.diag([0.3, 1.1]).astype(complex)
T = np.array([0.0, 0.2, 0.5])


def phases(t):
    return np.exp(-1j * np.diag(H).real * t)


@pytest.mark.parametrize("precision,scale", [("fp64", 1e-301), ("mixed", 1e-33)])
def test_small_master_equation_with_atol_zero(qt, precision, scale):
    """A matrix whose entries (none with a zero part) have subnormal weights."""
    mixed = precision == "mixed"
    X = scale * np.array([[1 + 2j, 1.5 - 1j], [2 + 1j, -1 + 1.5j]])
    o = qt.qt_opts_default(rtol=1e-6 if mixed else 1e-8, atol=0.0,
                           precision=qt.QT_MIXED if mixed else qt.QT_FP64)
    _, states, _ = qt.qt_mesolve(H, [], [], X, T, opts=o, store_states=True)
    for t, got in zip(T, states):
        want = phases(t)[:, None] * X * phases(t).conj()[None, :]
        assert np.abs(got - want).max() < (1e-5 if mixed else 1e-7) * scale


def test_trajectory_with_atol_zero(qt):
    psi = np.array([1 + 1j, 1e-301 * (1 + 1j)])
    O = np.array([[0, 1e300], [0, 0]], dtype=complex)
    o = qt.qt_opts_default(rtol=1e-8, atol=0.0)
    mean, _, _, _ = qt.qt_mcsolve(H, [], [O], psi, T, 1, opts=o)
    want = np.array([0.1 * phases(t)[0].conj() * phases(t)[1] for t in T])
    assert np.abs(mean[:, 0] - want).max() < 1e-8


def test_adjoint_with_atol_zero(qt):
    X = 1e-301 * np.array([[1 + 2j, 1.5 - 1j], [2 + 1j, -1 + 1.5j]])
    P1 = np.array([[1.0, 0.5], [0.5, 2.0]], dtype=complex)
    Z = np.zeros((2, 2), dtype=complex)
    adj = qt.Adjoint(H, np.diag([0.1, -0.2]).astype(complex), [], P1, Z, X, 2, 0.25, 1)
    om = torch.tensor([[0.5, -1.0]], dtype=torch.float64, device="cuda")
    ga = torch.zeros((1, 1), dtype=torch.float64, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    stb = torch.zeros(56, dtype=torch.uint8, device="cuda")
    adj.forward(om, ga, qt.qt_opts_default(rtol=1e-8, atol=0.0), loss, stats=stb)
    torch.cuda.synchronize()
    assert qt.stats_from_bytes(stb)["status"] == 0
    angle = np.diag(H).real * 0.5 + np.array([0.1, -0.2]) * 0.25 * (0.5 - 1.0)
    u = np.exp(-1j * angle)
    want = np.trace(P1 @ (u[:, None] * X * u.conj()[None, :])).real
    assert abs(loss.item() - want) < 1e-7 * 1e-301
