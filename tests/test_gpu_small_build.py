"""The pair build of small suspensions (all pairs tested, two launches) against
the oracle's pre-filter: sizes at the edges of its words, warps, staged
candidates and of its range, boxes with and without walls and periodic axes,
positions outside the box, particles with more partners than the grid build
has slots, and the capacity rule."""
import numpy as np
import pytest

import gen
import oracle

pytestmark = pytest.mark.gpu


def build(parts, dom, capacity, params=None):
    import torch

    import paper_1308_6482_gb300 as lub
    pl = lub.Pipeline(parts, dom, params or lub.default_params(), capacity=capacity)
    rc, cnt = lub.lub_pairs_build(pl.ctx.h, pl.P.c, pl.D, pl.prm, pl.pair_i, pl.pair_j, pl.cap, pl.d_count,
                                  h_count=True)
    torch.cuda.synchronize()
    m = min(cnt, capacity)
    return rc, cnt, pl.pair_i[:m].cpu().numpy(), pl.pair_j[:m].cpu().numpy(), pl


def scattered(n, seed, periodic, walls, spread=1.0):
    """n overlapping or touching spheroids in a box, some outside it."""
    rng = np.random.default_rng(seed)
    L = max(45.0, (n * 900.0) ** (1.0 / 3.0))
    sh = gen.aspect_shapes(n, rng)
    q = gen.random_quaternions(n, rng)
    p = dict(qw=q[:, 0].copy(), qx=q[:, 1].copy(), qy=q[:, 2].copy(), qz=q[:, 3].copy(),
             r_par=sh[:, 0].copy(), r_perp=sh[:, 1].copy())
    for k in "xyz":
        p[k] = L * (rng.random(n) * spread - 0.5 * (spread - 1.0))
    gen.velocities(p, rng)
    return p, dict(L=(L, L, L), periodic=periodic, walls=[(0.0, 1), (L, -1)][:walls])


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 256, 257, 1025, 1535, 1536, 1537, 4097])
@pytest.mark.parametrize("periodic,walls", [((True, True, True), 0), ((True, True, False), 2),
                                            ((False, False, False), 1)])
def test_lists_match_the_oracle(n, periodic, walls):
    parts, dom = scattered(n, 700 + n, periodic, walls, 3.0 if n % 2 else 1.0)
    opi, opj = oracle.candidates(parts, dom, 1.0)
    rc, cnt, pi, pj, _ = build(parts, dom, len(opi) + 64 * n)
    assert rc == 0 and cnt == len(opi)
    np.testing.assert_array_equal(pi, opi)
    np.testing.assert_array_equal(pj, opj)


def test_far_from_the_origin_and_on_the_cut_off():
    # coordinates a thousand boxes away, and spheres exactly at or within 2^-30 of the cut-off
    rng = np.random.default_rng(5)
    n = 300
    p = {k: np.zeros(n, np.float32) for k in ("qx", "qy", "qz")}
    p["qw"] = np.ones(n, np.float32)
    p["r_par"] = p["r_perp"] = np.full(n, 4.5, np.float32)
    idx = np.arange(n)
    p["x"] = 64.0 * 1024 + 40.0 * (idx // 2 % 10) + 10.0 * (idx % 2) + np.where(idx % 2, (idx % 3 - 1) * 2.0 ** -30, 0.0)
    p["y"] = -64.0 * 512 + 40.0 * (idx // 20)
    p["z"] = 20.0 * np.ones(n)
    gen.velocities(p, rng)
    dom = dict(L=(640.0, 1024.0, 64.0), periodic=(True, True, True), walls=[])
    opi, opj = oracle.candidates(p, dom, 1.0)
    rc, cnt, pi, pj, _ = build(p, dom, 4096)
    assert rc == 0 and 0 < cnt < n // 2
    np.testing.assert_array_equal(pi, opi)
    np.testing.assert_array_equal(pj, opj)


def test_more_partners_than_slots_and_the_capacity_rule():
    import paper_1308_6482_gb300 as lub
    rng = np.random.default_rng(8)
    n = 61
    p = {k: np.zeros(n, np.float32) for k in ("qx", "qy", "qz")}
    p["qw"] = np.ones(n, np.float32)
    p["r_par"] = p["r_perp"] = np.where(np.arange(n) == 0, 12.0, 0.8).astype(np.float32)
    k = np.arange(n)  # sixty small spheres on a Fibonacci sphere around a large one
    z = 1 - 2 * (k + 0.5) / n
    ph = k * np.pi * (3 - 5 ** 0.5)
    r = np.where(k == 0, 0.0, 13.2)
    p["x"], p["y"], p["z"] = 60 + r * np.sqrt(1 - z * z) * np.cos(ph), 60 + r * np.sqrt(1 - z * z) * np.sin(ph), 60 + r * z
    gen.velocities(p, rng)
    dom = dict(L=(120.0,) * 3, periodic=(True,) * 3, walls=[])
    opi, opj = oracle.candidates(p, dom, 1.0)
    assert (opi == 0).sum() == 60
    over = int(np.maximum(np.bincount(opi, minlength=n) - 16, 0).sum())
    rc, cnt, pi, pj, pl = build(p, dom, len(opi) + over)
    assert rc == 0 and cnt == len(opi)
    np.testing.assert_array_equal(pi, opi)
    np.testing.assert_array_equal(pj, opj)
    rc, cnt, _, _, pl = build(p, dom, len(opi) + over - 1)
    assert rc == lub.LUB_ERR_CAPACITY and cnt == len(opi) + over == pl.count()


def test_semi_axis_above_the_bound_is_an_argument_error():
    import paper_1308_6482_gb300 as lub
    parts, dom = scattered(40, 3, (True, True, True), 0)
    P = lub.DeviceParticles(parts, max_semi_axis=0.9 * float(max(parts["r_par"].max(), parts["r_perp"].max())))
    pl = lub.Pipeline(P, dom, lub.default_params(), capacity=2000)
    with pytest.raises(lub.LubError):
        pl.build_pairs()
    # the next build on the same context is clean
    ok = lub.Pipeline(parts, dom, lub.default_params(), capacity=2000, ctx=pl.ctx)
    assert ok.build_pairs() == len(oracle.candidates(parts, dom, 1.0)[0])
