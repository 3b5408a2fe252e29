"""The rigid sub-step's rotation at every size: half angles from 0 to far above
the 0.2 rad up to which its sine and cosine are series.  The update is in double
and rounded to single once (2^-24 of a quaternion's component or of a rate; the
double arithmetic's own error, some 1e-15 times the half angle, is far below)."""
import numpy as np
import pytest

import gen
import oracle
from parity import gpu_params

pytestmark = pytest.mark.gpu

HALF = [0.0, 1e-30, 1e-9, 1e-4, 0.05, 0.1999999, 0.2, 0.2000001, 0.25, 1.0, 3.0, 30.0]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("dt", [1.0, 0.125])
def test_half_angles_on_both_sides_of_the_series(prec, dt):
    import torch

    import paper_1308_6482_gb300 as lub
    rng = np.random.default_rng(8)
    n = 40 * len(HALF)
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    w = (2.0 / dt * np.repeat(HALF, 40)[:, None] * u).astype(np.float32)
    q = gen.random_quaternions(n, rng)
    sh = gen.aspect_shapes(n, rng)
    z = np.zeros(n)
    parts = dict(x=z, y=z.copy(), z=z.copy(), qw=q[:, 0].copy(), qx=q[:, 1].copy(), qy=q[:, 2].copy(), qz=q[:, 3].copy(),
                 r_par=sh[:, 0].copy(), r_perp=sh[:, 1].copy(), vx=z.astype(np.float32), vy=z.astype(np.float32),
                 vz=z.astype(np.float32), wx=w[:, 0].copy(), wy=w[:, 1].copy(), wz=w[:, 2].copy())
    dom = dict(L=(100.0, 100.0, 100.0), periodic=(False, False, False), walls=[])
    pl = lub.Pipeline(parts, dom, gpu_params(prec), capacity=1024)
    pl.force.zero_()
    pl.torque.zero_()
    pl.rigid_step(1.0, dt)
    torch.cuda.synchronize()
    got = {k: v.cpu().numpy().astype(np.float64) for k, v in pl.P.t.items()}
    ref = oracle.rigid_step(parts, np.zeros((n, 3)), np.zeros((n, 3)), 1.0, dt)
    for k in ("qw", "qx", "qy", "qz"):
        np.testing.assert_allclose(got[k], ref[k], rtol=0, atol=2.0 ** -24 + 1e-12, err_msg=k)
    size = np.linalg.norm(w.astype(np.float64), axis=1)
    for k in ("wx", "wy", "wz"):
        assert np.all(np.abs(got[k] - ref[k]) <= (2.0 ** -24 + 1e-12) * size * 3.0), k


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_rates_that_are_not_numbers_leave_the_orientation(prec):
    import torch

    import paper_1308_6482_gb300 as lub
    parts, dom, _, _ = gen.pair_stream(20, seed=61, kind="aspect")
    parts = {k: np.array(v) for k, v in parts.items()}
    parts["wx"][3] = parts["wz"][4] = np.nan
    pl = lub.Pipeline(parts, dom, gpu_params(prec), capacity=1024)
    pl.force.zero_()
    pl.torque.zero_()
    n = pl.n
    pl.torque[n + 7] = float("nan")   # the torque's y component on particle 7
    pl.rigid_step(1.0, 0.1)
    torch.cuda.synchronize()
    got = {k: v.cpu().numpy() for k, v in pl.P.t.items()}
    odd = np.array([3, 4, 7])
    for k in ("qw", "qx", "qy", "qz"):
        assert np.isfinite(got[k]).all()
        np.testing.assert_allclose(got[k][odd], parts[k][odd], rtol=0, atol=2.0 ** -23)
    for k in ("wx", "wy", "wz"):
        assert np.isnan(got[k][odd]).all() and np.isfinite(np.delete(got[k], odd)).all()
