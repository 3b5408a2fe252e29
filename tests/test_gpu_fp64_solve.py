"""Double-precision closest points: the result and the iteration count are
those of the FP64 Newton iteration (restated here in numpy), although the
library runs the iterations in FP32 and float-float: ordinary pairs, nearly
spherical and strongly overlapping ones, pairs whose line of centres is the
solution, warm starts far from, near to and at the solution, and small
iteration limits."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu


def newton_counts(parts, dom, pi, pj, maxit, start=None):
    """Iterations of the FP64 iteration: steps clamped to 0.5, halved where g falls, stop below 1e-7."""
    q = np.stack([parts[k].astype(np.float64) for k in ("qw", "qx", "qy", "qz")], 1)
    R = gen._rotmat(q)[:, :, 2]
    a, c = parts["r_perp"].astype(np.float64), parts["r_par"].astype(np.float64)
    pos = np.stack([parts[k] for k in "xyz"], 1)
    out = np.zeros(len(pi), int)
    for m, (i, j) in enumerate(zip(pi, pj)):
        if a[i] == c[i] and a[j] == c[j]:
            continue
        d = pos[j] - pos[i]
        dl = np.linalg.norm(d)
        n = d / dl
        if start is not None and 0.25 < start[m] @ start[m] < 4 and start[m] @ d > 0:
            n = start[m]
        n = n / np.linalg.norm(n)
        body = [(R[i], a[i] ** 2, c[i] ** 2 - a[i] ** 2), (R[j], a[j] ** 2, c[j] ** 2 - a[j] ** 2)]
        noise = 1e-14 * (dl + max(a[i], c[i]) + max(a[j], c[j]))
        e = np.array([1.0, 0, 0]) if abs(n[0]) < 0.6 else np.array([0, 1.0, 0])
        t1 = e - (e @ n) * n
        t1 /= np.linalg.norm(t1)
        acc, halvings = None, 0
        for it in range(maxit):
            t2 = np.cross(n, t1)
            g, g1, g2 = n @ d, t1 @ d, t2 @ d
            P = np.zeros((2, 2))
            A = 0.0
            for o, a2, ee in body:
                cc, u = o @ n, np.array([o @ t1, o @ t2])
                s = np.sqrt(a2 + ee * cc * cc)
                g -= s
                g1 -= ee * cc / s * u[0]
                g2 -= ee * cc / s * u[1]
                P += a2 / s * (np.eye(2) + ee / s ** 2 * np.outer(u, u))
                A += a2 / s
            P += g * np.eye(2)
            out[m] = it + 1
            if acc is not None and g < acc[0] - noise and halvings < 12:
                halvings += 1
                acc[1] *= 0.5
                n = acc[2] + acc[1][0] * acc[3] + acc[1][1] * acc[4]
                n /= np.linalg.norm(n)
                t1 = acc[3] - (acc[3] @ n) * n
                t1 /= np.linalg.norm(t1)
                continue
            det = P[0, 0] * P[1, 1] - P[0, 1] ** 2
            if P[0, 0] > 0 and det > 0:
                s = np.linalg.solve(P, [g1, g2])
            else:
                s = np.array([g1, g2]) / (abs(P[0, 0]) + abs(P[1, 1]) + abs(P[0, 1]) + A)
            sn = np.linalg.norm(s)
            if sn > 0.5:
                s *= 0.5 / sn
            acc = [g, s.copy(), n, t1, t2]
            n = n + s[0] * t1 + s[1] * t2
            n /= np.linalg.norm(n)
            t1 = t1 - (t1 @ n) * n
            t1 /= np.linalg.norm(t1)
            if sn < 1e-7:
                break
    return out


def solve(parts, dom, pi, pj, start=None, **kw):
    import torch

    import paper_1308_6482_gb300 as lub
    warm = "none" if start is None else "previous"
    pl = lub.Pipeline(parts, dom, lub.default_params(precision="fp64", warm_start=warm, **kw), capacity=len(pi))
    pl.set_pairs(pi, pj)
    if start is not None:
        pl.nrm.copy_(torch.as_tensor(np.ascontiguousarray(start.T).reshape(-1)))
    pl.closest()
    torch.cuda.synchronize()
    return pl.results()


def check(parts, dom, pi, pj, r, start=None, maxit=32):
    np.testing.assert_array_equal(r["iters"], newton_counts(parts, dom, pi, pj, maxit, start))
    ok = (r["status"] & 6) == 0
    cp = oracle.closest(parts, dom, pi[ok], pj[ok])
    assert np.abs(r["h"][ok] - cp["h"]).max(initial=0) <= 1e-12 * 40
    # the normal's error against the FP64 iteration's: both stop within about 1e-14 of the solution
    assert np.linalg.norm(r["n"][ok] - cp["n"], axis=1).max(initial=0) <= 1e-10
    return ok


@pytest.mark.parametrize("kind", ["aspect", "mixed"])
@pytest.mark.parametrize("maxit", [32, 4, 1])
def test_counts_and_results(kind, maxit):
    parts, dom, pi, pj = gen.pair_stream(700, seed=61, kind=kind, gap_range=(1e-4, 1.0))
    r = solve(parts, dom, pi, pj, max_newton=maxit)
    check(parts, dom, pi, pj, r, maxit=maxit)
    if maxit == 32:
        assert not np.any(r["status"])


def test_nearly_spherical_and_overlapping():
    parts, dom, pi, pj = gen.pair_stream(600, seed=62, kind="aspect", gap_range=(1e-4, 1.0))
    rng = np.random.default_rng(3)
    near = np.arange(1200) < 500
    parts["r_perp"] = np.where(near, parts["r_par"] * (1 + 1e-4 * rng.standard_normal(1200)), parts["r_perp"]).astype(np.float32)
    for k in "xyz":  # pushed together: overlaps up to a third of the distance
        parts[k] = parts[k].copy()
        parts[k][pj] -= 0.3 * (np.arange(600) % 3 == 0) * (parts[k][pj] - parts[k][pi])
    r = solve(parts, dom, pi, pj)
    check(parts, dom, pi, pj, r)


def test_solution_on_the_line_of_centres_and_warm_starts():
    parts, dom, pi, pj = gen.pair_stream(300, seed=63, kind="aspect", gap_range=(1e-3, 1.0))
    r = solve(parts, dom, pi, pj)
    rng = np.random.default_rng(4)
    for size in (0.0, 1e-9, 1e-7, 3e-6, 1e-3, 0.3):
        start = r["n"] + size * rng.standard_normal((300, 3))
        start *= rng.uniform(0.8, 1.2, (300, 1))
        w = solve(parts, dom, pi, pj, start=start)
        ok = check(parts, dom, pi, pj, w, start=start)
        assert ok.all()
    # pole to pole: the first step is zero
    for k in ("qx", "qy", "qz"):
        parts[k] = np.zeros(600, np.float32)
    parts["qw"] = np.ones(600, np.float32)
    for k in "xy":
        parts[k][pj] = parts[k][pi]
    parts["z"] = parts["z"].copy()
    parts["z"][pj] = parts["z"][pi] + parts["r_par"][pi] + parts["r_par"][pj] + 0.1
    w = solve(parts, dom, pi, pj)
    assert np.all(w["iters"] == 1) and np.abs(w["h"] - 0.1).max() <= 1e-6
