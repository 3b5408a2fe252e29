"""The link kernel at the edges of its batches (8 pairs per warp) and site
boxes of very different sizes, against the oracle's brute force."""
import numpy as np
import pytest

import gen
from test_gpu_links import check, lub, run  # noqa: F401  (lub: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 7, 8, 9, 15, 16, 17, 63, 65])
def test_batches_of_pairs_with_walls_and_invalid_pairs(lub, count):
    # a warp takes 8 pairs, a block 32; wall pairs, bad indices and self pairs among them give zeros
    parts, dom, pi, pj = gen.pair_stream(count, seed=90 + count, kind="mixed", gap_range=(0.02, 1.5))
    pi, pj = pi.copy(), pj.copy()
    bad = np.arange(count) % 5 == 3
    pj[bad] = np.where(np.arange(count)[bad] % 2 == 0, -1, pi[bad])
    qi, qj, F, T, nl = run(lub, parts, dom, pi, pj)
    assert not np.any(nl[bad]) and not np.any(F[bad]) and not np.any(T[bad])
    check(parts, dom, pi[~bad], pj[~bad], F[~bad], T[~bad], nl[~bad]) if (~bad).any() else None


def test_large_and_small_particles(lub):
    # boxes of thousands of sites beside boxes of a few
    parts, dom, pi, pj = gen.pair_stream(40, seed=97, kind="spheres", gap_range=(0.02, 1.0))
    for k in ("r_par", "r_perp"):
        parts[k] = parts[k].copy()
    a, b = pi, pj
    grow = np.where(np.arange(40) % 2 == 0, 3.0, 0.25)
    for k in ("x", "y", "z"):  # the pair scaled about its first centre
        parts[k] = parts[k].copy()
        parts[k][b] = parts[k][a] + (parts[k][b] - parts[k][a]) * grow
    for idx in (a, b):
        parts["r_par"][idx] = (parts["r_par"][idx] * grow).astype(np.float32)
        parts["r_perp"][idx] = parts["r_par"][idx]
    qi, qj, F, T, nl = run(lub, parts, dom, pi, pj)
    ref = check(parts, dom, pi, pj, F, T, nl)
    assert ref["links"].max() > 64
