"""lub_correct in one pass (mixed precision, small pair lists) against the
separate calls and the oracle: list lengths at the edges of warps and blocks,
and Newton tolerances at which none, some or all pairs are solved again in
FP64 (by the first lanes of their block), with walls and invalid pairs."""
import numpy as np
import pytest

import gen
from parity import compare, oracle_ref

pytestmark = pytest.mark.gpu


def both(parts, dom, pi, pj, **kw):
    import torch

    import paper_1308_6482_gb300 as lub
    out = []
    for fused in (True, False):
        pl = lub.Pipeline(parts, dom, lub.default_params(**kw), capacity=max(len(pi), 1) + 7)
        pl.set_pairs(pi, pj)
        if fused:
            pl.correct()
        else:
            pl.closest()
            pl.resistance()
            pl.apply()
        torch.cuda.synchronize()
        out.append(pl.results())
    return out


@pytest.mark.parametrize("count", [1, 31, 33, 63, 64, 65, 129, 3001])
@pytest.mark.parametrize("tol", [1e-4, 1.5e-7, 1e-12])
def test_one_pass_matches_the_calls_and_the_oracle(count, tol):
    parts, dom, pi, pj = gen.pair_stream(count, seed=500 + count, kind="aspect", gap_range=(1e-4, 1.0))
    one, sep = both(parts, dom, pi, pj, newton_tol=tol)
    # the same solves; both forms' contractions may differ by a rounding of the FP32 step
    same = one["status"] == sep["status"]
    assert same.mean() >= (1.0 if tol != 1.5e-7 else 0.98)
    if tol == 1e-12:
        assert np.all(one["status"] & 8)
    ref = oracle_ref(parts, dom, pi, pj)
    compare(parts, dom, one, ref, "mixed", pi, pj)
    sc = 30.0
    assert np.abs(one["h"] - sep["h"]).max() <= 1e-11 * sc
    assert np.abs(one["n"] - sep["n"]).max() <= 1e-11


def test_walls_and_invalid_pairs():
    parts, dom = gen.config_prolate_wall(seed=6)
    rng = np.random.default_rng(7)
    pi = rng.integers(0, 64, 300).astype(np.int32)
    pj = rng.integers(-3, 66, 300).astype(np.int32)  # walls 0, bad walls, bad indices, self pairs
    one, sep = both(parts, dom, pi, pj)
    np.testing.assert_array_equal(one["status"], sep["status"])
    np.testing.assert_array_equal(one["iters"], sep["iters"])
    assert np.abs(one["h"] - sep["h"]).max() <= 1e-9
    scale = np.abs(sep["force"]).max()
    assert np.abs(one["force"] - sep["force"]).max() <= 1e-4 * scale


@pytest.mark.parametrize("tol", [1e-4, 1e-12])
@pytest.mark.parametrize("capacity", [160000, 160001, 1600000, 1600001])
def test_forms_at_their_capacities(capacity, tol):
    """The one-pass kernel's two register budgets and the separate kernels for
    long lists are chosen by the pair arrays' capacity: the same list through
    each, next to the smallest capacity's results."""
    import torch

    import paper_1308_6482_gb300 as lub
    parts, dom, pi, pj = gen.pair_stream(1000, seed=77, kind="aspect", gap_range=(1e-4, 1.0))
    res = []
    for cap in (1000, capacity):
        pl = lub.Pipeline(parts, dom, lub.default_params(newton_tol=tol), capacity=cap)
        pl.set_pairs(pi, pj)
        pl.correct()
        torch.cuda.synchronize()
        res.append(pl.results())
    a, b = res
    compare(parts, dom, b, oracle_ref(parts, dom, pi, pj), "mixed", pi, pj)
    np.testing.assert_array_equal(a["status"], b["status"])
    np.testing.assert_array_equal(a["iters"], b["iters"])
    assert np.abs(a["h"] - b["h"]).max() <= 1e-11 * 30.0
    assert np.abs(a["n"] - b["n"]).max() <= 1e-11
