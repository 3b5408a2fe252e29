"""The pair list's own look-back (the kernel that scans the counts and writes the
list): a tile that never publishes, as if its block never ran, makes the tiles
after it poll to their bound.  The build returns, reports LUB_ERR_TIMEOUT
(through the host count and through lub_sync_status, which clears it), writes
nothing outside the list, and the next build on the same context is exact.  In
the test build of the library, in a child process."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys, time
sys.path.insert(0, ROOT)
import numpy as np
import torch
import gen
import paper_1308_6482_gb300 as lub
L = lub.load_library()
torch.cuda.set_device(0)
n, tiles = int(sys.argv[1]), int(sys.argv[2])
if n <= 40000:
    parts, dom = gen.config_mixed_suspension(N=n, phi=0.2, seed=12)
else:  # tiles of 1,024 particles from 262,144 on: spheres on a lattice, touching along x
    k = np.arange(n)
    side = 70
    parts = {f: np.zeros(n, np.float32) for f in ("qx", "qy", "qz", "vx", "vy", "vz", "wx", "wy", "wz")}
    parts["qw"] = np.ones(n, np.float32)
    parts["r_par"] = parts["r_perp"] = np.full(n, 1.0, np.float32)
    parts["x"], parts["y"], parts["z"] = 2.5 * (k % side) + 1.0, 4.0 * (k // side % side) + 1.0, 4.0 * (k // side ** 2) + 1.0
    dom = dict(L=(400.0, 400.0, 400.0), periodic=(False, False, False), walls=[(0.0, 1)])
pl = lub.Pipeline(parts, dom, lub.default_params())
m = pl.build_pairs()
ref = pl.pair_i[:m].cpu().numpy(), pl.pair_j[:m].cpu().numpy()
cap, pad = m + 5000, 4096
pi = torch.full((cap + pad,), -77, dtype=torch.int32, device="cuda")
pj = torch.full((cap + pad,), -77, dtype=torch.int32, device="cuda")

def build(h_count):
    pi.fill_(-77)
    pj.fill_(-77)
    t = time.time()
    try:
        rc, cnt = lub.lub_pairs_build(pl.ctx.h, pl.P.c, pl.D, pl.prm, pi, pj, cap, pl.d_count, h_count=h_count)
        torch.cuda.synchronize()
    except lub.LubError as e:
        rc, cnt = e.code, None
    return rc, cnt, time.time() - t

def status():
    try:
        lub.lub_sync_status(pl.ctx.h)
        return 0
    except lub.LubError as e:
        return e.code

out = []
for tile in (0, 3, tiles - 2):
    for h_count in (True, False):
        assert L.lub_test_mute_list_tile(tile) == 0
        rc, _, t = build(h_count)
        torch.cuda.synchronize()
        o = dict(tile=tile, h_count=h_count, rc=rc, s=t, status=[status(), status()])
        o["outside"] = bool((pi[m:] == -77).all()) and bool((pj[m:] == -77).all())
        assert L.lub_test_mute_list_tile(-1) == 0
        rc, cnt, _ = build(True)
        o["next"] = rc == 0 and cnt == m and np.array_equal(pi[:m].cpu().numpy(), ref[0]) and np.array_equal(
            pj[:m].cpu().numpy(), ref[1]) and status() == 0
        out.append(o)
print("RESULT " + json.dumps(out))
""".replace("ROOT", repr(ROOT))


@pytest.mark.parametrize("n,tile", [(5000, 256), (270000, 1024)])
def test_a_stalled_tile_of_the_list_is_reported(n, tile):
    import paper_1308_6482_gb300 as lub
    from paper_1308_6482_gb300 import build
    so = build.build(testing=True)
    r = subprocess.run([sys.executable, "-c", CHILD, str(n), str(-(-n // tile))], cwd=ROOT,
                       env=dict(os.environ, LUB_LIBRARY=so), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    out = json.loads([ln for ln in r.stdout.splitlines() if ln.startswith("RESULT ")][-1][7:])
    assert len(out) == 6
    for o in out:
        # without the host count the call only enqueues: the record is lub_sync_status's
        assert o["rc"] == (lub.LUB_ERR_TIMEOUT if o["h_count"] else 0), o
        assert o["status"] == [lub.LUB_ERR_TIMEOUT, 0], o
        assert o["s"] < 30.0 and o["outside"] and o["next"], o
