"""Links of thin discs: the extent of a disc seen nearly edge-on to its axis is
a small difference of large squares, and a lattice site just inside it still
counts.  Each pair has a site of i up to 3e-3 inside i's extreme point along an
axis and a sphere next to it; the links against the oracle's exactly, the
forces by the norm of each pair's force (its components may be differences of
much larger link forces)."""
import numpy as np
import pytest

import gen
import oracle
from helpers import make_parts, open_domain, quat_from_z_to
from test_gpu_links import MU, QBAR, lub, run  # noqa: F401  (lub: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rpar,rperp", [(0.0382, 100.0), (0.058, 100.0), (0.13, 100.0), (0.5, 100.0), (1.0, 30.0)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_sites_at_the_end_of_a_thin_disc(lub, rpar, rperp, axis):
    rng = np.random.default_rng(30 + axis)
    m = 64
    pos, q = np.zeros((2 * m, 3)), np.zeros((2 * m, 4))
    x = np.eye(3)[axis]
    rpar, rperp = float(np.float32(rpar)), float(np.float32(rperp))
    for k in range(m):
        o = x + rng.choice([0.0, 1e-4, 1e-3, 1e-2]) * rng.normal(size=3)
        # the axis of the quaternion as single precision holds it
        qk = quat_from_z_to(o / np.linalg.norm(o)).astype(np.float32).astype(np.float64)
        o = gen._rotmat(qk[None])[0, :, 2]
        sigma = np.sqrt(rperp ** 2 + (rpar ** 2 - rperp ** 2) * o[axis] ** 2)
        top = (rperp ** 2 * x + (rpar ** 2 - rperp ** 2) * o[axis] * o) / sigma
        site = np.array([1000.0, 1000.0, 1000.0]) * (k % 8 + 1)
        pos[2 * k] = site - top + rng.uniform(1e-5, 3e-3) * x
        pos[2 * k + 1] = site + 2.2 * x
        q[2 * k], q[2 * k + 1] = qk, (1, 0, 0, 0)
    a, b = np.tile([rpar, 1.6], m), np.tile([rperp, 1.6], m)
    v = 1e-3 * rng.normal(size=(2 * m, 6)).astype(np.float32)
    parts = make_parts(pos, q, a, b, v[:, :3], v[:, 3:])
    # the oracle gets what the library holds in single precision
    parts = {key: (u if key in "xyz" else u.astype(np.float32)) for key, u in parts.items()}
    i = np.arange(0, 2 * m, 2, dtype=np.int32)
    _, _, F, T, nl = run(lub, parts, open_domain(), i, i + 1)
    ref = oracle.links(parts, open_domain(), i, i + 1, MU, QBAR)
    np.testing.assert_array_equal(nl, ref["links"])
    size = np.linalg.norm(ref["F"], axis=1)
    assert np.all(np.linalg.norm(F - ref["F"], axis=1) <= 1e-9 * size)
    assert np.all(np.linalg.norm(T - ref["T"], axis=1) <= 1e-9 * size * rperp)
    assert (ref["links"] > 0).mean() > 0.9
