"""Double-precision closest points of cold lists on either side of the lengths
between which the FP64 iteration runs alone: iteration counts, statuses, normals
and gaps of the same pairs in lists of every kind."""
import numpy as np
import pytest

import gen
from test_gpu_fp64_solve import check, solve

pytestmark = pytest.mark.gpu

FROM, TO = 512, 24576


@pytest.mark.parametrize("kind", ["aspect", "mixed"])
def test_the_same_pairs_in_lists_of_every_length(kind):
    parts, dom, pi, pj = gen.pair_stream(TO + 1, seed=44, kind=kind, gap_range=(1e-4, 1.0))
    runs = [solve(parts, dom, pi[:m], pj[:m]) for m in (TO + 1, TO, FROM, FROM - 1)]
    for r in runs[1:]:
        m = len(r["h"])
        np.testing.assert_array_equal(r["iters"], runs[0]["iters"][:m])
        np.testing.assert_array_equal(r["status"], runs[0]["status"][:m])
        # both end on a step below 1e-7 from the same solution, squared by Newton
        assert np.linalg.norm(r["n"] - runs[0]["n"][:m], axis=1).max() <= 1e-12
        assert np.abs(r["h"] - runs[0]["h"][:m]).max() <= 1e-12
    for r in runs[2:]:
        m = len(r["h"])
        assert check(parts, dom, pi[:m], pj[:m], r).all()
