"""The cell-grid pair build at the edges that small inputs were made for.  Single
suspensions of up to 1,536 particles take the all-pairs build, so the inputs of
those tests are run on the grid here: the same tests with their suspension as
the one member of an ensemble (which always takes the grid), and the same
configurations repeated or enlarged beyond 1,536 particles."""
import numpy as np
import pytest

import gen
import oracle
import test_gpu_parity as parity_tests
from parity import compare, oracle_ref, run_gpu
from test_gpu_parity import crowded_particle
from test_zz_no_alloc import _static_vs_context

pytestmark = pytest.mark.gpu
SMALL = 1536

AS_A_MEMBER = [(f, dict(prec=p)) for f in ("test_more_partners_than_slots",
                                           "test_more_partners_than_slots_on_the_filters_edge",
                                           "test_candidates_on_the_filters_edge_beyond_the_buffer",
                                           "test_candidates_exactly_on_the_list_cutoff") for p in ("fp64", "mixed")]
AS_A_MEMBER += [("test_small_periodic_boxes_list_every_pair_once", dict(L=v)) for v in (9.5, 11.5, 14.5)]
AS_A_MEMBER += [("test_open_box_with_particles_outside_it", dict(shift=v)) for v in ((0.0, 0.0, 0.0), (-0.3, 0.25, -0.1))]
AS_A_MEMBER += [("test_dense_packings", dict(case="five_cells")), ("test_candidates_at_the_list_cutoff", dict(P=500)),
                ("test_wall_pairs_at_the_list_cutoff", {})]


@pytest.mark.parametrize("name,args", AS_A_MEMBER)
def test_as_the_one_member_of_an_ensemble(name, args, monkeypatch):
    import paper_1308_6482_gb300 as lub

    class Member(lub.Pipeline):
        def __init__(self, parts, dom, *a, **kw):
            P = lub.DeviceParticles(parts, batch_offsets=np.array([0, len(parts["x"])], np.int32))
            super().__init__(P, [dom], *a, **kw)

    monkeypatch.setattr(lub, "Pipeline", Member)
    getattr(parity_tests, name)(**args)


def repeated(parts, dom, k, shift):
    """k^3 copies, a multiple of `shift` apart, in a box of k shifts a side."""
    n = len(parts["x"])
    out = {f: np.tile(np.asarray(v), k ** 3) for f, v in parts.items()}
    c = np.repeat(np.arange(k ** 3), n)
    for a, f in enumerate("xyz"):
        out[f] = out[f] + shift * (c // k ** a % k)
    return out, dict(dom, L=(shift * k,) * 3)


def check(parts, dom, prec):
    assert len(parts["x"]) > SMALL
    pi, pj = oracle.candidates(parts, dom, 1.0)
    g = run_gpu(parts, dom, prec)
    np.testing.assert_array_equal(g["pi"], pi)
    np.testing.assert_array_equal(g["pj"], pj)
    compare(parts, dom, g, oracle_ref(parts, dom, pi, pj), prec, pi, pj)
    return pi, pj


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("gap", [0.5, 1.0 - 2e-5])
def test_many_particles_of_more_partners_than_slots(prec, gap):
    # 64 clusters of 31: beyond the slots, on the overflow list (gap 0.5) or, with more than 15 candidates
    # inside the FP32 margin in one warp, from the buffer of decided candidates (gap at the cut-off)
    import paper_1308_6482_gb300 as lub
    parts, dom = repeated(*crowded_particle(gap=gap), 4, 64.0)
    pi, pj = check(parts, dom, prec)
    assert np.sum(pi == 0) == 30
    if gap == 0.5:
        over = int(np.maximum(np.bincount(pi, minlength=len(parts["x"])) - 16, 0).sum())
        pl = lub.Pipeline(parts, dom, lub.default_params(), capacity=len(pi) + over - 1)
        rc, need = lub.lub_pairs_build(pl.ctx.h, pl.P.c, pl.D, pl.prm, pl.pair_i, pl.pair_j, pl.cap, pl.d_count,
                                       h_count=True)
        assert rc == lub.LUB_ERR_CAPACITY and need == len(pi) + over
        pl2 = lub.Pipeline(parts, dom, lub.default_params(), capacity=need)
        assert pl2.build_pairs() == len(pi)
        np.testing.assert_array_equal(pl2.results()["pj"], pj)


def test_partners_beyond_the_slots_from_the_second_decision():
    # 377,177 particles (all rows of a slot in one warp, 1,024 particles a tile of the list): 12,167 clusters at
    # the cut-off, some 30 candidates inside the FP32 margin per warp, which decides 15 itself
    import torch

    import paper_1308_6482_gb300 as lub
    one = crowded_particle(gap=1.0 - 2e-5)
    ci, cj = oracle.candidates(*one, 1.0)
    n1, k = len(one[0]["x"]), 23
    parts, dom = repeated(*one, k, 64.0)
    at = n1 * np.arange(k ** 3)[:, None]
    pl = lub.Pipeline(parts, dom, lub.default_params(), capacity=16 * len(parts["x"]))
    assert pl.build_pairs() == len(ci) * k ** 3
    torch.cuda.synchronize()
    m = len(ci) * k ** 3
    np.testing.assert_array_equal(pl.pair_i[:m].cpu().numpy(), (at + ci).ravel())
    np.testing.assert_array_equal(pl.pair_j[:m].cpu().numpy(), (at + cj).ravel())


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_more_candidates_on_the_filters_edge_than_the_buffer_holds(prec):
    # a cubic lattice of 13^3 spheres, every neighbour inside the FP32 margin (listed along x and z)
    n, R = 13, 2.0
    a = np.array([2 * R + 1.0 - 2e-5, 2 * R + 1.0 + 2e-5, 2 * R + 1.0 - 2e-5])
    i = np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)
    rng = np.random.default_rng(9)
    q = gen.random_quaternions(len(i), rng)
    r = np.full(len(i), R, np.float32)
    parts = dict(zip("xyz", ((i + 0.5) * a).T.copy()), qw=q[:, 0].copy(), qx=q[:, 1].copy(), qy=q[:, 2].copy(),
                 qz=q[:, 3].copy(), r_par=r, r_perp=r.copy())
    gen.velocities(parts, rng)
    pi, _ = check(parts, dict(L=tuple(float(v) for v in n * a), periodic=(True, True, True), walls=[]), prec)
    assert len(pi) == 2 * len(i)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_pairs_exactly_on_the_cut_off_and_one_bit_beside_it(prec):
    # 900 sphere pairs at 2 R + Delta_L = 5, and 2^-30 nearer or farther (exactly representable)
    m = 900
    k = np.arange(m)
    base = np.stack([16.0 * (k % 30) + 8.0, 16.0 * (k // 30) + 8.0, 16.0 + 0.0 * k], 1)
    off = np.array([0.0, 2.0 ** -30, -(2.0 ** -30)])[k % 3]
    other = base.copy()
    other[k, k // 3 % 3] += 5.0 + off
    pos = np.stack([base, other], 1).reshape(-1, 3)
    # (unturned: the half-widths are then exactly 2 in any order of operations)
    q = np.tile(np.array([1, 0, 0, 0], np.float32), (2 * m, 1))
    r = np.full(2 * m, 2.0, np.float32)
    parts = dict(x=pos[:, 0].copy(), y=pos[:, 1].copy(), z=pos[:, 2].copy(), qw=q[:, 0].copy(), qx=q[:, 1].copy(),
                 qy=q[:, 2].copy(), qz=q[:, 3].copy(), r_par=r, r_perp=r.copy())
    gen.velocities(parts, np.random.default_rng(12))
    pi, pj = check(parts, dict(L=(480.0, 480.0, 480.0), periodic=(True, True, True), walls=[]), prec)
    np.testing.assert_array_equal(pi, 2 * k[off <= 0])


@pytest.mark.parametrize("shift", [(0.0, 0.0, 0.0), (-0.3, 0.25, -0.1)])
def test_open_box_with_particles_outside_it(shift):
    rng = np.random.default_rng(31)
    parts, dom = gen.suspension(gen.aspect_shapes(1800, rng), (130.0,) * 3, periodic=(False,) * 3, attach_prob=0.8,
                                seed=32)
    for k, f in zip("xyz", shift):
        parts[k] = parts[k] + f * 130.0
    check(parts, dom, "mixed")


def test_wall_pairs_on_the_cut_off():
    rng = np.random.default_rng(91)
    n, L = 2000, 1200.0
    a, b = rng.uniform(2.0, 8.0, (2, n)).astype(np.float32)
    q = gen.random_quaternions(n, rng)
    oz = gen._rotmat(q.astype(np.float64))[:, 2, 2]
    sz = np.sqrt(b.astype(float) ** 2 + (a.astype(float) ** 2 - b.astype(float) ** 2) * oz ** 2)
    k = np.arange(n)
    parts = dict(x=(k % 45 + 0.5) * (L / 45), y=(k // 45 + 0.5) * (L / 45), z=sz + 1.0 + rng.uniform(-1e-4, 1e-4, n),
                 qw=q[:, 0].copy(), qx=q[:, 1].copy(), qy=q[:, 2].copy(), qz=q[:, 3].copy(), r_par=a, r_perp=b)
    gen.velocities(parts, rng)
    pi, pj = check(parts, dict(L=(L, L, L), periodic=(True, True, False), walls=[(0.0, 1)]), "fp64")
    assert 0.25 * n < np.sum(pj < 0) < 0.75 * n


def test_static_build_clears_what_the_build_before_left():
    import torch

    import paper_1308_6482_gb300 as lub
    torch.cuda.set_device(0)
    for n, seed in ((32768, 2), (2000, 3), (5000, 4)):
        assert n > SMALL and _static_vs_context(lub, *gen.config_mixed_suspension(N=n, phi=0.25, seed=seed)) > n // 2
