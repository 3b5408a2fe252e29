"""The library's own FP64 scalar functions (logarithm, reciprocal, reciprocal
root, conversions on the integer pipe) against numpy, over the ranges they are
used in and at the ends of the exponent's range: through a hook of the test
build of the library, in a child process.

Bounds, from the operations' roundings (u = 2^-53): the reciprocal ends in one
multiply-add on a correction below 2^-22 (2 u), the root in one whose
correction carries the rounding of a y (4 u); the logarithm has a reciprocal,
four products and sums and, for k != 0, ln 2 rounded once (8 u, relative).
The conversions are exact or defined by their rounding."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53

CHILD = r"""
import ctypes, sys
sys.path.insert(0, ROOT)
import numpy as np
import torch
import paper_1308_6482_gb300 as lub
L = lub.load_library()
vp = ctypes.c_void_p
L.lub_test_math.restype = ctypes.c_int
L.lub_test_math.argtypes = [ctypes.c_int32, vp, vp, ctypes.c_int32, vp]
d = np.load(sys.argv[1])
out = {}
for fn, key in enumerate(("log1p", "rcp", "rsqrt", "widen", "round", "narrow")):
    x = torch.as_tensor(d[key], device="cuda")
    y = torch.empty_like(x)
    assert L.lub_test_math(fn, x.data_ptr(), y.data_ptr(), x.numel(), None) == 0
    torch.cuda.synchronize()
    out[key] = y.cpu().numpy()
np.savez(sys.argv[2], **out)
""".replace("ROOT", repr(ROOT))


def inputs():
    rng = np.random.default_rng(11)
    n = 20000
    sign = lambda v: np.where(rng.random(len(v)) < 0.5, -v, v)
    edge = np.array([np.sqrt(0.5), np.sqrt(2.0), 0.5, 1.0])
    edge = np.concatenate([np.nextafter(edge, 0), edge, np.nextafter(edge, 9)]) - 1
    bits = rng.integers(0, 1 << 32, n, dtype=np.uint32)
    with np.errstate(all="ignore"):
        f = bits.view(np.float32).astype(np.float64)
    sub = (rng.integers(0, 1 << 23, 2000).astype(np.uint32)).view(np.float32).astype(np.float64)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.0, -1.0])
    wide = sign(np.ldexp(1.0 + rng.random(n), rng.integers(-300, 300, n)))
    near = sign(np.ldexp(1.0 + rng.random(n), rng.integers(-152, 130, n)))
    ties = sign((1 + rng.integers(0, 1 << 23, 2000) * 2.0 ** -23 + 2.0 ** -24) * 2.0 ** rng.integers(-40, 40, 2000))
    return dict(
        log1p=np.concatenate([-1 + 10.0 ** rng.uniform(-15, 0, n), -10.0 ** rng.uniform(-18, 0, n),
                              10.0 ** rng.uniform(-18, 3, n), edge, [-1.0, -1.5, np.nan, np.inf, 0.0, -1e-300]]),
        rcp=sign(np.concatenate([np.ldexp(1.0 + rng.random(n), rng.integers(-1022, 1021, n)),
                                 2.0 ** np.arange(-1022, 1022), [2.0 ** -1022]])),
        rsqrt=np.concatenate([np.ldexp(1.0 + rng.random(n), rng.integers(-1022, 1024, n)),
                              2.0 ** np.arange(-1022, 1024)]),
        widen=np.concatenate([f, sub, -sub, special]),
        round=np.concatenate([wide, near, ties, special]),
        narrow=np.concatenate([wide, near, special]))


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    from paper_1308_6482_gb300 import build
    so = build.build(testing=True)
    d = tmp_path_factory.mktemp("math")
    x = inputs()
    np.savez(d / "x.npz", **x)
    r = subprocess.run([sys.executable, "-c", CHILD, str(d / "x.npz"), str(d / "y.npz")], cwd=ROOT,
                       env=dict(os.environ, LUB_LIBRARY=so), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return x, dict(np.load(d / "y.npz"))


def within(y, ref, bound):
    """|y - ref| <= bound |ref|, ref a long double; non-finite values equal."""
    ref = np.asarray(ref)
    fin = np.isfinite(ref.astype(np.float64))
    np.testing.assert_array_equal(y[~fin], ref[~fin].astype(np.float64))
    err = np.abs(y[fin].astype(np.longdouble) - ref[fin])
    assert np.all(err <= bound * np.abs(ref[fin])), float((err / np.maximum(np.abs(ref[fin]), 1e-300)).max() / U)


# (on a host without long doubles the reference itself carries some u)
SLACK = 0 if np.finfo(np.longdouble).nmant > 52 else 2


def test_logarithm(results):
    x, y = results[0]["log1p"], results[1]["log1p"]
    with np.errstate(all="ignore"):
        ref = np.log1p(x.astype(np.longdouble))
    within(y, ref, (8 + SLACK) * U)


def test_reciprocal_and_root(results):
    x, y = results
    within(y["rcp"], 1 / x["rcp"].astype(np.longdouble), (2 + SLACK) * U)
    within(y["rsqrt"], 1 / np.sqrt(x["rsqrt"].astype(np.longdouble)), (4 + SLACK) * U)


def test_conversions(results):
    x, y = results
    np.testing.assert_array_equal(y["widen"], x["widen"])
    num = ~np.isnan(x["widen"])
    np.testing.assert_array_equal(np.signbit(y["widen"])[num], np.signbit(x["widen"])[num])
    with np.errstate(all="ignore"):
        ref = x["round"].astype(np.float32).astype(np.float64)
    np.testing.assert_array_equal(y["round"], ref)
    # truncated to 24 bits within the normal float range, 0 below it, infinite above it
    v, t = x["narrow"], y["narrow"]
    a = np.abs(v)
    ok = (a >= 2.0 ** -126) & (a < 2.0 ** 128)
    assert np.all(np.abs(t[ok]) <= a[ok]) and np.all(a[ok] - np.abs(t[ok]) < np.ldexp(1.0, np.frexp(a[ok])[1] - 24))
    assert np.all(np.sign(t[ok]) == np.sign(v[ok]))
    assert np.all(t[a < 2.0 ** -126] == 0) and np.all(np.isinf(t[(a >= 2.0 ** 128) | np.isnan(a)]))
