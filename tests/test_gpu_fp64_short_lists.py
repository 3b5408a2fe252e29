"""Double-precision closest points of short lists (two warps per 32 pairs) and of
longer ones: the same pairs give the same bits, iteration counts and statuses in
either, walls, spheres and invalid pairs among them, from cold and warm starts
and at small iteration limits."""
import numpy as np
import pytest

import gen
from test_gpu_fp64_solve import check, solve

pytestmark = pytest.mark.gpu

# longest arrays of the short form, longest list that takes two warps per 32 pairs
SHORT, TWO = 24576, 9728


@pytest.mark.parametrize("kind", ["aspect", "mixed"])
@pytest.mark.parametrize("maxit", [32, 4, 1])
@pytest.mark.parametrize("warm", [False, True])
def test_the_same_pairs_in_short_and_long_lists(kind, maxit, warm):
    parts, dom, pi, pj = gen.pair_stream(SHORT + 1, seed=44, kind=kind, gap_range=(1e-4, 1.0))
    dom = dict(dom, walls=[(float(parts["z"].min()) - 20.0, 1)], periodic=(dom["periodic"][0], dom["periodic"][1], False))
    pj = pj.copy()
    odd = np.arange(len(pi)) % 37
    pj[odd == 5] = -1                 # walls
    pj[odd == 11] = pi[odd == 11]     # invalid
    start = None
    if warm:
        d = np.stack([parts[k][np.maximum(pj, 0)] - parts[k][pi] for k in "xyz"], 1)
        d /= np.maximum(np.linalg.norm(d, axis=1, keepdims=True), 1e-9)
        start = d + 0.1 * np.random.default_rng(3).normal(size=d.shape)
    runs = {m: solve(parts, dom, pi[:m], pj[:m], start[:m] if warm else None, max_newton=maxit)
            for m in (SHORT + 1, SHORT, TWO + 1, TWO, 2048, 2047, 513, 128, 127, 33, 1)}
    ref = runs[SHORT + 1]
    for m, r in runs.items():
        for f in ("n", "h", "iters", "status"):
            np.testing.assert_array_equal(r[f], ref[f][:m], err_msg="%s of %d" % (f, m))
    ok = (odd[:513] != 5) & (odd[:513] != 11)
    r = {f: v[ok] for f, v in runs[513].items() if f in ("n", "h", "iters", "status")}
    check(parts, dom, pi[:513][ok], pj[:513][ok], r, start[:513][ok] if warm else None, maxit)


@pytest.mark.parametrize("capacity", [SHORT, SHORT + 1])
def test_the_autotuner_keeps_the_default_where_the_shape_is_fixed(capacity):
    import paper_1308_6482_gb300 as lub
    parts, dom = gen.config_mixed_suspension(N=1000, phi=0.25, seed=4)
    pl = lub.Pipeline(parts, dom, lub.default_params(precision="fp64"), capacity=capacity)
    shape = pl.autotune(reps=1)["closest_fp64"]
    assert shape == (64, 256) if capacity <= SHORT else shape[0] in (64, 128)
