"""The deterministic sums, bitwise against the same additions on the host in
the order of (pair, side): particles of 0 to 100 entries (the rounds of eight,
the sort by rank up to 32 and in place beyond it), entries on either side, pairs
in shuffled order, walls among them; the forms by eight lanes and by one lane a
particle on either side of the rule between them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ENTRIES = [0, 1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 100]


def pair_list(n, extra, rng):
    """Particle k < len(ENTRIES) in ENTRIES[k] pairs, on both sides, with partners
    among the rest; `extra` more pairs of the rest; every eleventh a wall's."""
    k = np.repeat(np.arange(len(ENTRIES)), ENTRIES)
    other = rng.integers(len(ENTRIES), n, len(k))
    side = rng.random(len(k)) < 0.5
    pi, pj = np.where(side, other, k), np.where(side, k, other)
    a = rng.integers(len(ENTRIES), n, extra)
    b = rng.integers(len(ENTRIES), n - 1, extra)
    b = np.where(b >= a, b + 1, b)
    b = np.where(np.arange(extra) % 11 == 3, -1, b)
    pi, pj = np.concatenate([pi, a]), np.concatenate([pj, b])
    o = rng.permutation(len(pi))
    return pi[o].astype(np.int32), pj[o].astype(np.int32)


# one lane a particle below 1.5 entries each from 131,072 particles on and 3.5 from 250,000
@pytest.mark.parametrize("n,extra", [(40, 0), (9001, 30000), (20000, 20000), (131071, 40000), (131072, 40000),
                                     (131072, 110000), (249999, 300000), (250000, 300000), (250000, 500000)])
@pytest.mark.parametrize("accumulate", [0, 1])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_sums_in_the_order_of_pairs_and_sides(n, extra, accumulate, prec):
    import torch

    import paper_1308_6482_gb300 as lub
    rng = np.random.default_rng(n + extra)
    pi, pj = pair_list(n, extra, rng)
    m = len(pi)
    dt = np.float32 if prec == "mixed" else np.float64
    # levers of zero: the contributions are +-(F, T) exactly, the order of the additions is all that is left
    FT = (rng.normal(size=(6, m)) * 10.0 ** rng.uniform(-3, 3, (6, m))).astype(dt)
    was = rng.normal(size=(2, 3 * n)).astype(dt)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    force, torque = dev(was[0]), dev(was[1])
    ctx = lub.Context()
    args = (dev(pi), dev(pj), dev(np.array([m], np.int32)), m, dev(FT.reshape(-1)),
            torch.zeros(6 * m, dtype=torch.float32 if prec == "mixed" else torch.float64, device="cuda"))
    prm = lub.default_params(precision=prec)
    lub.lub_apply(ctx.h, *args, n, force, torque, prm.precision, accumulate, 1)
    torch.cuda.synchronize()
    idx = np.stack([pi, pj], 1).reshape(-1)
    keep = idx >= 0
    for got, rows, old in ((force, FT[:3], was[0]), (torque, FT[3:], was[1])):
        for c in range(3):
            v = np.stack([rows[c], -rows[c]], 1).reshape(-1)
            ref = np.zeros(n, dt)
            np.add.at(ref, idx[keep], v[keep])
            if accumulate:
                ref = old.reshape(3, n)[c] + ref
            np.testing.assert_array_equal(got.cpu().numpy().reshape(3, n)[c], ref)
