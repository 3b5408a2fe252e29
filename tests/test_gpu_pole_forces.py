"""FP64 forces where the normal is close to a particle's symmetry axis: the
contact lies next to a pole, where the direction away from the axis is what
cancellation leaves of the contact point's offset.  Spheroids lying flat on or
standing up at a wall, and coaxial pairs, tilted by 1e-2 down to 1e-11 rad,
through all three calls that evaluate the resistance, against the oracle."""
import numpy as np
import pytest

import oracle
from helpers import axis_angle_quat, make_parts, open_domain
from parity import compare, oracle_ref

pytestmark = pytest.mark.gpu

TILTS = np.array([1e-2, 1e-3, 1e-5, 1e-7, 1e-8, 1e-9, 1e-10, 1e-11])
SHAPES = {"prolate": (6.0, 3.0), "oblate": (3.0, 6.0), "needle": (12.0, 2.0), "disc": (1.5, 9.0)}
GAPS = np.array([0.02, 0.3, 0.55])


def tilted(rng, angle):
    ph = rng.uniform(0, 2 * np.pi)
    return axis_angle_quat([np.cos(ph), np.sin(ph), 0.0], angle)


def velocities(rng, n):
    return rng.normal(size=(n, 3)).astype(np.float32), rng.normal(size=(n, 3)).astype(np.float32)


def as_f32(parts):
    return {k: (v if k in "xyz" else np.asarray(v, np.float32)) for k, v in parts.items()}


def at_wall(shape, seed):
    """One spheroid per (tilt, gap), 50 apart, over a wall at z = 0."""
    rng = np.random.default_rng(seed)
    a, b = SHAPES[shape]
    t, h = [v.ravel() for v in np.meshgrid(TILTS, GAPS)]
    n = len(t)
    k = np.arange(n)
    q = np.array([tilted(rng, v) for v in t])
    v, w = velocities(rng, n)
    parts = make_parts(np.stack([50.0 * k, 0.0 * k, 0.0 * k], 1), q, np.full(n, a), np.full(n, b), v, w)
    parts = as_f32(parts)
    oz = 1 - 2 * (parts["qx"].astype(float) ** 2 + parts["qy"].astype(float) ** 2)
    parts["z"] = np.sqrt(b * b + (a * a - b * b) * oz * oz) + h
    dom = open_domain()
    dom["walls"] = [(0.0, 1)]
    return parts, dom, k.astype(np.int32), np.full(n, -1, np.int32)


def coaxial(shape, seed):
    """Two spheroids one above the other, tilts of the same order, a little off line."""
    rng = np.random.default_rng(seed)
    a, b = SHAPES[shape]
    t, h = [v.ravel() for v in np.meshgrid(TILTS, GAPS)]
    m = len(t)
    pos, q = np.zeros((2 * m, 3)), np.zeros((2 * m, 4))
    for k in range(m):
        q[2 * k], q[2 * k + 1] = tilted(rng, t[k]), tilted(rng, 0.4 * t[k])
        pos[2 * k] = (60.0 * k, 0.0, 0.0)
        pos[2 * k + 1] = pos[2 * k] + (0.3 * t[k], -0.2 * t[k], 2 * a + h[k])
    v, w = velocities(rng, 2 * m)
    parts = as_f32(make_parts(pos, q, np.full(2 * m, a), np.full(2 * m, b), v, w))
    i = np.arange(0, 2 * m, 2, dtype=np.int32)
    return parts, open_domain(), i, i + 1


@pytest.mark.parametrize("call", ["resistance", "resistance_apply", "correct"])
@pytest.mark.parametrize("config", [at_wall, coaxial])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_forces_next_to_a_pole(shape, config, call):
    import torch

    import paper_1308_6482_gb300 as lub
    parts, dom, pi, pj = config(shape, 3)
    pl = lub.Pipeline(parts, dom, lub.default_params(precision="fp64"), capacity=len(pi))
    pl.set_pairs(pi, pj)
    if call == "correct":
        pl.correct()
    else:
        pl.closest()
        if call == "resistance":
            pl.resistance()
            pl.apply()
        else:
            pl.resistance_apply()
    torch.cuda.synchronize()
    ref = oracle_ref(parts, dom, pi, pj)
    assert (ref["pf"]["status"] & (oracle.ST_NOCONV | oracle.ST_DEGENERATE) == 0).all()
    compare(parts, dom, pl.results(), ref, "fp64", pi, pj)
