"""The work that users of the lubrication library have it do, as cases for timing.

Each case goes through the public Python entry points of the package, on
inputs made here from a seed alone (torch, on the GPU when there is one):

  step      one correction step of a suspension (``Pipeline.step``): the pair
            build, closest points, resistance and scatter
  ensemble  the same step over many independent suspensions in one call
  calls     the step as separate calls with the deterministic force sum
  temporal  the step with the paper's temporal warm start: the previous
            list's normals carried over to the new list
  substeps  one lattice-Boltzmann step of particle motion: new poses, the pair
            list, then ten sub-steps of forces and rigid motion with contacts
  links     the link-based lubrication of Ding and Aidun on a pair list
  closest   closest points of given pairs from the learned warm start
  train     one training step of the learned warm start (gradients and Adam)

``exact`` gives what a case returns in 64-bit torch arithmetic, written here
from the method's formulas.
"""
import math

import numpy as np
import torch

import paper_1308_6482_gb300 as lub
from paper_1308_6482_gb300._lib import LUB_MLP_PARAMS, LUB_MLP_WORK_PER_SAMPLE, lub_mlp_adam, lub_mlp_forward_backward
from paper_1308_6482_gb300.mlp import SHAPES, WarmStartMLP

DELTA_L = 1.0                     # list cut-off (Sec. III A)
SUB_DT = 0.02                     # sub-step (stable for contacts at h_c = 0.01 and these masses)
PI = math.pi


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # a first small suspension over a wall (the paper's smallest runs):
        # 64 prolates in a 42^3 box, called eagerly; launches and host time
        {"name": "wall_64", "kind": "step", "n": 64, "shape": "prolate", "phi": 0.195, "box": "wall",
         "precision": "mixed", "per_pair": True, "graph": False},
        # the mixed suspension (spheres and oblates, log-uniform gaps), the
        # step captured once in a CUDA graph as a time loop does
        {"name": "mixed_32k", "kind": "step", "n": 32768, "shape": "mixed", "phi": 0.3, "box": "periodic",
         "precision": "mixed", "per_pair": True, "graph": True},
        # the large dense run between two walls: a million spheroids
        {"name": "dense_1m", "kind": "step", "n": 1048576, "shape": "aspect", "phi": 0.5, "box": "slit",
         "precision": "mixed", "per_pair": True, "graph": True},
        # a parameter study: independent suspensions of many sizes and
        # volume fractions advanced together
        {"name": "ensemble_256k", "kind": "ensemble", "members": 96, "n": 262144, "graph": True},
        # double precision, an odd size, only the sums wanted (a reference run)
        {"name": "fp64_20k", "kind": "step", "n": 20011, "shape": "aspect", "phi": 0.45, "box": "periodic",
         "precision": "fp64", "per_pair": False, "graph": False},
        # bitwise reproducible sums: separate calls, ragged size
        {"name": "calls_100k", "kind": "calls", "n": 100003, "shape": "aspect", "phi": 0.4, "box": "periodic"},
        # time stepping with the temporal warm start
        {"name": "temporal_131k", "kind": "temporal", "n": 131072, "shape": "aspect", "phi": 0.5, "box": "slit"},
        # ten particle sub-steps per lattice-Boltzmann step, contacts on
        {"name": "substeps_32k", "kind": "substeps", "n": 32768, "shape": "mixed", "phi": 0.3, "sub": 10},
        # the comparison model on the mixed suspension's pairs
        {"name": "links_32k", "kind": "links", "n": 32768, "shape": "mixed", "phi": 0.3},
        # fresh pairs (no previous step) from the learned start, both precisions
        {"name": "learned_fp64_128k", "kind": "closest", "pairs": 131072, "precision": "fp64"},
        {"name": "learned_mixed_1m", "kind": "closest", "pairs": 1048576, "precision": "mixed"},
        # training the learned start: the shipped weights' batch
        {"name": "train_8192", "kind": "train", "batch": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "ensemble", "calls", "temporal", "substeps", "links", "closest", "train"])
    if kind == "step":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        n = _log_int(rng, 48, 700000 if precision == "mixed" else 60000)
        return {"kind": kind, "n": n, "shape": rng.choice(["aspect", "mixed", "prolate"]),
                "phi": round(rng.uniform(0.1, 0.5), 3), "box": rng.choice(["periodic", "wall", "slit"]),
                "precision": precision, "per_pair": precision == "mixed", "graph": rng.random() < 0.5}
    if kind == "ensemble":
        members = _log_int(rng, 2, 200)
        return {"kind": kind, "members": members, "n": members * _log_int(rng, 300, 2500), "graph": rng.random() < 0.5}
    if kind in ("calls", "temporal"):
        return {"kind": kind, "n": _log_int(rng, 500, 200000), "shape": rng.choice(["aspect", "mixed"]),
                "phi": round(rng.uniform(0.15, 0.5), 3), "box": rng.choice(["periodic", "slit"])}
    if kind == "substeps":
        return {"kind": kind, "n": _log_int(rng, 200, 32768), "shape": rng.choice(["mixed", "aspect"]),
                "phi": round(rng.uniform(0.15, 0.4), 3), "sub": rng.randint(2, 10)}
    if kind == "links":
        return {"kind": kind, "n": _log_int(rng, 200, 24000), "shape": rng.choice(["mixed", "aspect"]),
                "phi": round(rng.uniform(0.15, 0.4), 3)}
    if kind == "closest":
        precision = rng.choice(["mixed", "fp64"])
        return {"kind": kind, "pairs": _log_int(rng, 100, 1000000 if precision == "mixed" else 120000),
                "precision": precision}
    return {"kind": "train", "batch": _log_int(rng, 64, 8192)}


def _pairs_estimate(case):
    """Listed pairs per particle grow linearly with the volume fraction."""
    return case["n"] * max(0.05, 8.65 * case.get("phi", 0.3) - 0.065)


def work(case):
    """Bytes read and written once, and the formulas' operations (a step in
    mixed precision counts a float-float operation as ten)."""
    kind = case["kind"]
    if kind == "train":
        nb, p = case["batch"], LUB_MLP_PARAMS
        return {"bytes": nb * (12 + 4 + 4 + 1) * 4 + p * 4 * 8, "flops": 6.0 * nb * (12 * 128 + 128 * 128 + 128 * 4)}
    if kind == "closest":
        m = case["pairs"]
        its = 170.0 * (3.0 if case["precision"] == "fp64" else 2.2)
        gap = 240.0 if case["precision"] == "fp64" else 2400.0
        return {"bytes": m * (2 * 48 + 8 + 33), "flops": m * (its + gap + 36864.0)}
    m = _pairs_estimate(case)
    if kind == "links":
        return {"bytes": case["n"] * 72.0 + m * (8 + 76), "flops": m * 150000.0}
    fp64 = case.get("precision") == "fp64"
    per_pair = 170.0 * (4.2 if fp64 else 3.6) + (240.0 if fp64 else 2400.0) + 1300.0
    out = 8 + 24 + (58 if case.get("per_pair", True) else 0)
    sub = case.get("sub", 1)
    return {"bytes": case["n"] * (72.0 + (48 if fp64 else 24)) + m * out, "flops": m * per_pair * sub}


# ---------------------------------------------------------------------------
# inputs: shapes and packings
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt=0):
    g = torch.Generator(device=_device())
    g.manual_seed((int(seed) * 1000003 + salt * 7919 + 17) & 0x7FFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=_device(), dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=_device(), dtype=torch.float64)


def _shapes(kind, shape, g):
    """(r_par, r_perp): prolates (6, 3), half spheres 4.5 and half oblates
    (3, 6), or aspect ratios log-uniform in [1/3, 3] at equivalent radius 4.5."""
    u = _rand(g, *shape)
    if kind == "prolate":
        a, b = torch.full_like(u, 6.0), torch.full_like(u, 3.0)
    elif kind == "mixed":
        a, b = torch.where(u < 0.5, 4.5, 3.0).double(), torch.where(u < 0.5, 4.5, 6.0).double()
    else:
        lam = torch.exp((2 * u - 1) * math.log(3.0))
        a, b = 4.5 * lam ** (2.0 / 3.0), 4.5 * lam ** (-1.0 / 3.0)
    return a.float().double(), b.float().double()  # the values that single precision holds


def _rmax(kind):
    return {"prolate": 6.0, "mixed": 6.0, "aspect": 4.5 * 3.0 ** (2.0 / 3.0)}[kind]


def _volume(a, b):
    return 4.0 / 3.0 * PI * a * b * b


def _quat(g, *shape):
    q = _randn(g, *shape, 4)
    return (q / q.norm(dim=-1, keepdim=True)).float().double()


def _axis(q):
    w, x, y, z = q.unbind(-1)
    s = 2.0 / (w * w + x * x + y * y + z * z)
    return torch.stack([s * (x * z + w * y), s * (y * z - w * x), 1 - s * (x * x + y * y)], -1)


def _rotate(q, v):
    """exp(v / 2) q, normalised (lab-frame rotation vector v)."""
    a = v.norm(dim=-1, keepdim=True)
    s = torch.where(a > 0, torch.sin(0.5 * a) / a.clamp_min(1e-300), torch.full_like(a, 0.5))
    w, r = torch.cos(0.5 * a), s * v
    qw, qv = q[..., :1], q[..., 1:]
    p = torch.cat([w * qw - (r * qv).sum(-1, keepdim=True), w * qv + qw * r + torch.linalg.cross(r, qv)], -1)
    return p / p.norm(dim=-1, keepdim=True)


def _image(d, L, per):
    """Minimum image along the periodic axes."""
    return d - torch.where(per, L * torch.floor(d / L + 0.5), torch.zeros_like(d))


def _half_width(o, a2, e, n):
    """sigma(n) of a spheroid a2 I + e o o^T along unit n, and o.n."""
    c = (o * n).sum(-1)
    return torch.sqrt(a2 + e * c * c), c


def _neighbours(pos, reach, L, per, k):
    """Indices [B, n, k] of each particle's nearest particles by centre
    distance less both reaches (itself excluded)."""
    B, n, _ = pos.shape
    k = min(k, n - 1)
    out = torch.empty(B, n, k, dtype=torch.long, device=pos.device)
    rows = max(1, min(n, int(4e7) // (n * B)))
    for s in range(0, n, rows):
        e = min(n, s + rows)
        d2 = torch.zeros(B, e - s, n, device=pos.device, dtype=torch.float32)
        for a in range(3):
            d = pos[:, s:e, None, a].float() - pos[:, None, :, a].float()
            d = d - torch.where(per[..., a, None, None], L[:, a, None, None] * torch.round(d / L[:, a, None, None]), 0.0).float()
            d2 += d * d
        gap = d2.sqrt_() - reach[:, s:e, None].float() - reach[:, None, :].float()
        gap[:, torch.arange(e - s), torch.arange(s, e)] = float("inf")
        out[:, s:e] = gap.topk(k, dim=-1, largest=False, sorted=False).indices
    return out.sort(-1).values


def _gather(v, nb):
    """v [B, n, ...] at the neighbour indices [B, n, k]."""
    B, n, k = nb.shape
    f = v.reshape(B, n, -1)
    return torch.gather(f, 1, nb.reshape(B, n * k, 1).expand(-1, -1, f.shape[-1])).reshape(B, n, k, *v.shape[2:])


def _ascend(n, d, oi, a2i, ei, oj, a2j, ej):
    """One under-relaxed ascent step of g(n) = n.d - sigma_i - sigma_j on the
    sphere; g is a lower bound of the distance for every n."""
    si, ci = _half_width(oi, a2i, ei, n)
    sj, cj = _half_width(oj, a2j, ej, n)
    r = d - (a2i / si + a2j / sj)[..., None] * n - (ei * ci / si)[..., None] * oi - (ej * cj / sj)[..., None] * oj
    g = (n * r).sum(-1)
    t = r - g[..., None] * n
    curv = torch.maximum(a2i / si, a2i * (a2i + ei) / si ** 3) + torch.maximum(a2j / sj, a2j * (a2j + ej) / sj ** 3)
    m = n + t / (g + curv).clamp_min(1.0)[..., None]
    return m / m.norm(dim=-1, keepdim=True), g


def _pack(a, b, L, walls, g, sweeps=320):
    """Growth packing of B boxes [B, 3] at once (periodic, but for z where it is
    confined to [0, L_z] by walls): random placement, growth from half size
    to 2 % beyond full size with overlaps pushed apart, sizes reset.  Returns
    positions, quaternions and which particles touch no other (the rest, if
    any, are left out)."""
    B, n = a.shape
    dev = a.device
    per = torch.ones(B, 3, dtype=torch.bool, device=dev)
    per[:, 2] = ~walls
    pos = _rand(g, B, n, 3) * L[:, None, :]
    q = _quat(g, B, n)
    rmax = torch.maximum(a, b)
    Lk, pk = L[:, None, None, :], per[:, None, None, :]
    nb = nrm = reach = None
    for t in range(sweeps + 1):
        last = t == sweeps
        s = 1.0 if last else min(1.02, 0.5 + 0.52 * t / (0.7 * sweeps))
        a2, e = (s * b) ** 2, (s * a) ** 2 - (s * b) ** 2
        if t % 16 == 0 or last:
            nb = _neighbours(pos, rmax, L, per, 64 if last else 40)
            reach = 1.02 * (_gather(rmax, nb) + rmax[..., None])
        a2j, ej = _gather(a2, nb), _gather(e, nb)
        o = _axis(q)
        oj = _gather(o, nb)
        d = _image(_gather(pos, nb) - pos[:, :, None, :], Lk, pk)
        oi = o[:, :, None, :].expand_as(d)
        a2i, ei = a2[..., None].expand_as(a2j), e[..., None].expand_as(ej)
        if t % 16 == 0 or last:
            nrm = d / d.norm(dim=-1, keepdim=True).clamp_min(1e-9)
            for _ in range(24 if last else 3):
                nrm, gap = _ascend(nrm, d, oi, a2i, ei, oj, a2j, ej)
        nrm, gap = _ascend(nrm, d, oi, a2i, ei, oj, a2j, ej)
        # bounding spheres apart: no contact (whose nearest image may change)
        r = d.norm(dim=-1)
        away = r > reach + 0.1
        nrm = torch.where(away[..., None], d / r.clamp_min(1e-9)[..., None], nrm)
        gap = torch.where(away, r - reach, gap)
        wz, _ = _half_width(o, a2, e, torch.tensor([0.0, 0.0, 1.0], device=dev, dtype=torch.float64))
        lo = torch.where(walls[:, None], pos[..., 2] - wz, torch.full_like(wz, 1e9))
        hi = torch.where(walls[:, None], L[:, 2, None] - pos[..., 2] - wz, torch.full_like(wz, 1e9))
        if last:
            keep = (lo > 1e-3) & (hi > 1e-3)
            # of each overlapping pair the one of larger index goes
            bad = (gap < 1e-3) & (nb < torch.arange(n, device=dev)[None, :, None])
            keep &= ~bad.any(-1)
            pos = pos - torch.where(per[:, None], L[:, None] * torch.floor(pos / L[:, None]), torch.zeros_like(pos))
            return pos, q, keep, nb, nrm, gap
        push = (0.02 - gap).clamp_min(0.0)
        si, ci = _half_width(oi, a2i, ei, nrm)
        rho = (a2i / si)[..., None] * nrm + (ei * ci / si)[..., None] * oi
        f = push[..., None] * nrm
        pos = pos - 0.45 * f.sum(2)
        spin = torch.linalg.cross(rho, f).sum(2) / (rmax * rmax)[..., None]
        q = _rotate(q, -0.6 * spin)
        pos[..., 2] += (0.02 - lo).clamp_min(0.0) - (0.02 - hi).clamp_min(0.0)


def _close_gaps(pos, q, keep, nb, nrm, gap, g):
    """Mutual nearest neighbours moved together along their common normal, to
    gaps log-uniform in [1e-4, 1] (only closer, and only where no third
    particle is met): translation along the normal keeps the closest points."""
    B, n, k = nb.shape
    dead = ~_gather(keep, nb)
    gg = torch.where(dead, torch.full_like(gap, 1e9), gap)
    best, slot = gg.min(-1)
    mate = torch.gather(nb, 2, slot[..., None])[..., 0]
    mutual = keep & (torch.gather(mate, 1, mate) == torch.arange(n, device=pos.device)[None])
    u = _rand(g, B, n)
    target = torch.exp(math.log(1e-4) * torch.minimum(u, torch.gather(u, 1, mate)))
    move = 0.5 * (best - target).clamp_min(0.0)
    move = torch.where(mutual, torch.minimum(move, torch.gather(move, 1, mate)), torch.zeros_like(move))
    # every other neighbour farther than both sides move
    others = torch.where(torch.arange(k, device=pos.device) == slot[..., None], torch.full_like(gg, 1e9), gg)
    ok = mutual & (others - _gather(move, nb) > move[..., None]).all(-1)
    ok &= torch.gather(ok, 1, mate)
    step = torch.gather(nrm, 2, slot[..., None, None].expand(-1, -1, 1, 3))[..., 0, :]
    # both sides of a pair use the smaller index's normal, so that they move oppositely
    first = torch.arange(n, device=pos.device)[None] < mate
    other = -torch.gather(step, 1, mate[..., None].expand(-1, -1, 3))
    step = torch.where(first[..., None], step, other)
    return pos + torch.where(ok[..., None], move[..., None] * step, torch.zeros_like(step))


def _best(keep, n):
    """The first n kept particles (overlapping ones only where too few are left)."""
    return torch.argsort(~keep, stable=True)[:n].sort().values


_WALLS = {"periodic": 0, "wall": 1, "slit": 2}


def _suspension(case, seed):
    """Particles (float64 tensors) and the domain of a one-suspension case: a
    packing of at most 16,384 particles tiled along x and y, each tile moved
    and turned by small random amounts of its own."""
    n, kind, box = case["n"], case["shape"], case.get("box", "periodic")
    g = _gen(seed, 1)
    k = -(-n // 16384)
    kx = int(math.ceil(math.sqrt(k)))
    ky = -(-k // kx)
    n0 = -(-n // (kx * ky))
    n0 += 4 + n0 // 25  # a few more than needed: those left overlapping go
    a, b = _shapes(kind, (1, n0), g)
    side = (float(_volume(a, b).sum()) * kx * ky / case["phi"]) ** (1.0 / 3.0)
    side = max(side, 2.0 * (2 * _rmax(kind) + DELTA_L) * 1.02 * max(kx, 1))
    L0 = torch.tensor([[side / kx, side / ky, side]], dtype=torch.float64, device=a.device)
    walls = torch.tensor([box != "periodic"], device=a.device)
    pos, q, keep, nb, nrm, gap = _pack(a, b, L0, walls, g)
    if kind == "mixed":
        pos = _close_gaps(pos, q, keep, nb, nrm, gap, g)
    at = _best(keep[0], -(-n // (kx * ky)))
    pos, q, a, b = pos[0, at], q[0, at], a[0, at], b[0, at]
    if kx * ky > 1:
        m = len(at)
        sh = torch.tensor([[i * side / kx, j * side / ky, 0.0] for i in range(kx) for j in range(ky)],
                          dtype=torch.float64, device=pos.device)
        pos = (pos[None] + sh[:, None]).reshape(-1, 3)
        q, a, b = q.repeat(kx * ky, 1), a.repeat(kx * ky), b.repeat(kx * ky)
        if kind != "mixed":
            pos = pos + 0.002 * _randn(g, m * kx * ky, 3)
            q = _rotate(q, 0.0002 * _randn(g, m * kx * ky, 3))
    if len(pos) > n:
        at = torch.randperm(len(pos), generator=g, device=pos.device)[:n].sort().values
        pos, q, a, b = pos[at], q[at], a[at], b[at]
    order = torch.randperm(len(pos), generator=g, device=pos.device) if kind == "mixed" else None
    if order is not None:
        pos, q, a, b = pos[order], q[order], a[order], b[order]
    dom = {"L": (side, side, side), "periodic": (True, True, box == "periodic"),
           "walls": [(0.0, 1), (side, -1)][:_WALLS[box]]}
    return _parts(pos, q, a, b, g), dom


def _parts(pos, q, a, b, g):
    v = (1e-3 * _randn(g, len(pos), 6)).float().double()
    q = q.float().double()
    return {"pos": pos, "q": q, "a": a, "b": b, "v": v[:, :3].contiguous(), "w": v[:, 3:].contiguous()}


def _ensemble(case, seed):
    """Independent periodic suspensions back to back: packings of a few
    hundred spheroids at volume fractions in [0.1, 0.5], tiled k^3 times."""
    g = _gen(seed, 2)
    members, n = case["members"], case["n"]
    bases = min(members, 8)
    n0 = max(150, min(600, n // members))
    phi = 0.1 + 0.4 * (torch.arange(bases, device=_device(), dtype=torch.float64) + _rand(g, bases)) / bases
    a, b = _shapes("aspect", (bases, n0 + 4 + n0 // 25), g)
    side = (_volume(a, b).sum(1) / phi) ** (1.0 / 3.0)
    side = side.clamp_min(2.0 * (2 * _rmax("aspect") + DELTA_L) * 1.02)
    pos, q, keep, _, _, _ = _pack(a, b, side[:, None].expand(-1, 3).contiguous(),
                                  torch.zeros(bases, dtype=torch.bool, device=a.device), g)
    # sizes log-uniform over a factor of thirty about n / members, as k^3 copies
    size = torch.exp(3.4 * (torch.arange(members, device=a.device) + 0.5) / members)
    size = size / size.sum() * n
    k = (size / n0).pow(1.0 / 3.0).round().clamp(1, 6).long()
    k = k[torch.randperm(members, generator=g, device=a.device)].cpu().tolist()
    side_h, out, doms, offs = side.cpu().tolist(), [], [], [0]
    for m in range(members):
        c, km = m % bases, k[m]
        at = _best(keep[c], n0)
        r = torch.arange(km, device=a.device, dtype=torch.float64) * side_h[c]
        sh = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
        p = (pos[c, at][None] + sh[:, None]).reshape(-1, 3)
        p = p + 0.002 * _randn(g, len(p), 3)
        t = len(sh)
        out.append(_parts(p, q[c, at].repeat(t, 1), a[c, at].repeat(t), b[c, at].repeat(t), g))
        doms.append({"L": (side_h[c] * km,) * 3, "periodic": (True, True, True), "walls": []})
        offs.append(offs[-1] + len(p))
    parts = {key: torch.cat([o[key] for o in out]) for key in out[0]}
    return parts, doms, np.asarray(offs, np.int32)


def _fresh_pairs(m, seed):
    """Independent pairs at gaps log-uniform in [1e-4, 1] times the smallest
    semi-axis, each far from all others (no previous step to start from)."""
    g = _gen(seed, 3)
    a, b = _shapes("aspect", (2 * m,), g)
    q = _quat(g, 2 * m)
    o = _axis(q)
    a2, e = b * b, a * a - b * b
    n = _randn(g, m, 3)
    n = n / n.norm(dim=-1, keepdim=True)
    h = torch.exp(math.log(1e-4) * _rand(g, m)) * torch.minimum(a, b).reshape(m, 2).min(1).values

    def reach(k, v):
        s, c = _half_width(o[k::2], a2[k::2], e[k::2], v)
        return (a2[k::2] / s)[:, None] * v + (e[k::2] * c / s)[:, None] * o[k::2]

    side = int(math.ceil(m ** (1.0 / 3.0)))
    i = torch.arange(m, device=a.device)
    grid = torch.stack([i % side, (i // side) % side, i // (side * side)], 1).double()
    ra = (grid + 0.5) * 42.0 + 2 * _rand(g, m, 3) - 1
    rb = ra + reach(0, n) + h[:, None] * n + reach(1, n)
    pos = torch.stack([ra, rb], 1).reshape(2 * m, 3)
    dom = {"L": (side * 42.0,) * 3, "periodic": (False, False, False), "walls": []}
    return _parts(pos, q, a, b, g), dom


def _host(parts):
    """The package's particle dict (numpy) of the tensors above."""
    d = {}
    for keys, t in ((("x", "y", "z"), parts["pos"]), (("qw", "qx", "qy", "qz"), parts["q"]),
                    (("vx", "vy", "vz"), parts["v"]), (("wx", "wy", "wz"), parts["w"])):
        for c, key in enumerate(keys):
            d[key] = t[:, c].cpu().numpy().astype(np.float64 if key in "xyz" else np.float32)
    d["r_par"] = parts["a"].cpu().numpy().astype(np.float32)
    d["r_perp"] = parts["b"].cpu().numpy().astype(np.float32)
    return d


def _moved(parts, seed):
    """The next time step's poses."""
    g = _gen(seed, 4)
    p = dict(parts)
    p["pos"] = parts["pos"] + 0.01 * _randn(g, len(parts["pos"]), 3)
    p["q"] = _rotate(parts["q"], 0.005 * _randn(g, len(parts["pos"]), 3)).float().double()
    return p


def _train_inputs(case, seed):
    g = _gen(seed, 5)
    nb = case["batch"]
    x = _randn(g, nb, 12).float()
    t = (0.3 * torch.tanh(_randn(g, 12, 4).T @ x.double().T).T + 0.05 * _randn(g, nb, 4)).float()
    w = torch.cos(1.2 * _randn(g, nb, 4)).square().float()
    w[:, 0::2] = 1.0
    p = []
    for key, sh in SHAPES:
        scale = math.sqrt(2.0 / sh[1]) if key.startswith("W") else 0.05
        p.append((scale * _randn(g, *sh)).reshape(-1))
    p = torch.cat(p).float()
    # moments of a run some hundred steps old
    m = (1e-3 * _randn(g, len(p))).float()
    v = (1e-2 * (0.5 + _rand(g, len(p)))).square().float()
    return x, t.contiguous(), w.contiguous(), p, m, v


ADAM_T, ADAM_LR = 400, 1e-3


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _room(case):
    """Pairs that the arrays have room for, from the volume fraction."""
    if case["kind"] == "ensemble":
        return 6 * case["n"] + 1024
    return int(1.3 * case["n"] * (8.65 * case["phi"] + 0.4)) + 1024


def _views(pl, per_pair, iters=True):
    """The step's outputs: the sums and the pair arrays."""
    c, n = pl.cap, max(pl.n, 1)
    out = {"force": pl.force.view(3, n), "torque": pl.torque.view(3, n), "pair_i": pl.pair_i, "pair_j": pl.pair_j,
           "n": pl.nrm.view(3, c)}
    if per_pair:
        out.update(gap=pl.gap, status=pl.status, FT=pl.FT.view(6, c), lever=pl.lever.view(6, c))
        if iters:
            out["iters"] = pl.iters
    return out


def _pipeline(P, dom, prm, case):
    """A pipeline with its pair list built and zeros behind the last pair."""
    pl = lub.Pipeline(P, dom, prm, capacity=_room(case))
    for t in (pl.pair_i, pl.pair_j, pl.nrm, pl.gap, pl.status, pl.iters, pl.FT, pl.lever):
        t.zero_()
    m = pl.build_pairs(grow=False)
    assert m <= pl.cap, "more pairs than the arrays have room for"
    return pl


def _captured(call, graph):
    """The call itself, or its replay from a CUDA graph captured once."""
    call()
    if not graph:
        return call
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g.replay


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, w, p, m, v = _train_inputs(case, seed)
        ctx = lub.Context()
        nb = case["batch"]
        grads = torch.zeros_like(p)
        scratch = torch.empty(nb * LUB_MLP_WORK_PER_SAMPLE, device=x.device)
        rows = torch.empty(nb, device=x.device)

        def call():
            lub_mlp_forward_backward(ctx.h, p, x, t, w, nb, grads, scratch, rows)
            lub_mlp_adam(ctx.h, p, grads, m, v, LUB_MLP_PARAMS, ADAM_T, ADAM_LR)

        return {"call": call, "out": {"grads": grads, "loss": rows, "params": p, "m": m, "v": v}}

    if kind == "closest":
        parts, dom = _fresh_pairs(case["pairs"], seed)
        m = case["pairs"]
        prm = lub.default_params(precision=case["precision"], warm_start="mlp_all")
        pl = lub.Pipeline(lub.DeviceParticles(_host(parts)), dom, prm, capacity=m)
        WarmStartMLP.load().install(pl.ctx)
        pl.set_pairs(np.arange(0, 2 * m, 2), np.arange(1, 2 * m, 2))

        def call():
            lub.lub_closest_points(pl.ctx.h, pl.P.c, pl.D, pl.prm, pl.pair_i, pl.pair_j, pl.d_count, pl.cap, pl.nrm,
                                   pl.gap, pl.status)

        return {"call": call, "out": {"n": pl.nrm.view(3, m), "gap": pl.gap, "status": pl.status}}

    if kind == "ensemble":
        parts, doms, offs = _ensemble(case, seed)
        P = lub.DeviceParticles(_host(parts), batch_offsets=offs)
        pl = _pipeline(P, doms, lub.default_params(), case)
        return {"call": _captured(lambda: pl.step(form="fused"), case["graph"]), "out": _views(pl, True),
                "keep": pl}

    parts, dom = _suspension(case, seed)
    if kind == "substeps":
        P = lub.DeviceParticles(_host(parts), packed=True)
        pl = _pipeline(P, dom, lub.default_params(h_c=0.01, eps_c=100.0), case)
        poses = P.blob.clone()

        def call():
            P.blob.copy_(poses)  # the step's poses and velocities, handed over in one packed copy
            pl.substeps(case["sub"], 1.0, SUB_DT, form="fused")

        # what the host code takes back: forces, poses and velocities
        out = {key: t for key, t in _views(pl, False).items() if key != "n"}
        out.update({key: P.t[key] for key in ("x", "y", "z", "qw", "qx", "qy", "qz", "vx", "vy", "vz", "wx", "wy", "wz")})
        return {"call": _captured(call, True), "out": out, "keep": (pl, poses)}

    if kind == "links":
        pl = _pipeline(lub.DeviceParticles(_host(parts)), dom, lub.default_params(), case)
        f, t, c = pl.links()

        def call():
            pl.links()

        return {"call": call, "out": {"force": f.view(3, pl.cap), "torque": t.view(6, pl.cap), "links": c}}

    if kind == "temporal":
        # the previous step's list and normals, then the poses of this step
        prev = _pipeline(lub.DeviceParticles(_host(parts)), dom, lub.default_params(), case)
        prev.step(build=False, form="fused")
        prev.keep_previous()
        prm = lub.default_params(warm_start="previous")
        pl = _pipeline(lub.DeviceParticles(_host(_moved(parts, seed))), dom, prm, case)
        pl.prev_i, pl.prev_j, pl.prev_n = prev.prev_i, prev.prev_j, prev.prev_n
        pl.prev_count, pl.prev_cap = prev.prev_count, prev.prev_cap

        def call():
            pl.build_pairs(sync_count=False, grow=False)
            pl.carry()
            pl.correct()

        return {"call": call, "out": _views(pl, True)}

    if kind == "calls":
        pl = _pipeline(lub.DeviceParticles(_host(parts)), dom, lub.default_params(), case)
        return {"call": lambda: pl.step(deterministic=1), "out": _views(pl, True)}

    pl = _pipeline(lub.DeviceParticles(_host(parts)), dom, lub.default_params(precision=case["precision"]), case)
    per_pair = case["per_pair"]
    return {"call": _captured(lambda: pl.step(form="fused", per_pair=per_pair), case["graph"]),
            "out": _views(pl, per_pair), "keep": pl}


def run(state):
    state["call"]()
    return state["out"]


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _candidates(parts, dom):
    """The pair list (i, j, canonical order, walls last as j = -1 - w)."""
    pos, o = parts["pos"], _axis(parts["q"])
    a, b = parts["a"], parts["b"]
    dev, n = pos.device, len(pos)
    L = torch.tensor(dom["L"], dtype=torch.float64, device=dev)
    per = torch.tensor(dom["periodic"], device=dev)
    rmax = torch.maximum(a, b)
    a2, e = b * b, a * a - b * b
    edge = 2 * float(rmax.max()) + DELTA_L
    nc = [max(1, int(v // (edge * 1.0001))) for v in dom["L"]]
    p = pos - torch.where(per, L * torch.floor(pos / L), torch.zeros_like(pos))
    c = torch.stack([(p[:, k] / dom["L"][k] * nc[k]).floor().long().clamp(0, nc[k] - 1) for k in range(3)], 1)
    cell = (c[:, 2] * nc[1] + c[:, 1]) * nc[0] + c[:, 0]
    order = cell.argsort(stable=True)
    start = torch.searchsorted(cell[order].contiguous(), torch.arange(nc[0] * nc[1] * nc[2] + 1, device=dev))
    keys = []
    shifts = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)]
    block = 262144
    for sh in shifts:
        for s in range(0, n, block):
            i = torch.arange(s, min(n, s + block), device=dev)
            cc, ok = [], torch.ones(len(i), dtype=torch.bool, device=dev)
            for k in range(3):
                v = c[i, k] + sh[k]
                if dom["periodic"][k]:
                    v = v % nc[k]
                else:
                    ok &= (v >= 0) & (v < nc[k])
                    v = v.clamp(0, nc[k] - 1)
                cc.append(v)
            other = (cc[2] * nc[1] + cc[1]) * nc[0] + cc[0]
            cnt = torch.where(ok, start[other + 1] - start[other], 0)
            ii = torch.repeat_interleave(i, cnt)
            first = torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
            j = order[torch.repeat_interleave(start[other], cnt) + torch.arange(len(ii), device=dev) - first]
            up = ii < j
            ii, j = ii[up], j[up]
            d = _image(pos[j] - pos[ii], L, per)
            r = d.norm(dim=-1)
            near = r <= rmax[ii] + rmax[j] + DELTA_L
            ii, j, d, r = ii[near], j[near], d[near], r[near]
            nn = d / r[:, None]
            si, _ = _half_width(o[ii], a2[ii], e[ii], nn)
            sj, _ = _half_width(o[j], a2[j], e[j], nn)
            good = (r - si <= rmax[j] + DELTA_L) & (r - sj <= rmax[ii] + DELTA_L)
            keys.append(ii[good] * n + j[good])
    key = torch.unique(torch.cat(keys))
    i, j = key // n, key % n
    wz, _ = _half_width(o, a2, e, torch.tensor([0.0, 0.0, 1.0], device=dev, dtype=torch.float64))
    listed_walls = []
    for w, (z, s) in enumerate(dom["walls"]):
        k = torch.nonzero(s * (pos[:, 2] - z) - wz < DELTA_L)[:, 0]
        listed_walls.append(k * 2 + w)
    if listed_walls:
        k = torch.cat(listed_walls).sort().values
        i, j = torch.cat([i, k // 2]), torch.cat([j, -1 - k % 2])
    return i, j


def _side(t, k):
    """t at the indices k, at 0 where k names a wall."""
    return t[k.clamp_min(0)]


def _closest(parts, dom, i, j):
    """Normals and gaps by Newton's method on the sphere in 64 bits."""
    pos, o = parts["pos"], _axis(parts["q"])
    a2, e = parts["b"] ** 2, parts["a"] ** 2 - parts["b"] ** 2
    L = torch.tensor(dom["L"], dtype=torch.float64, device=pos.device)
    per = torch.tensor(dom["periodic"], device=pos.device)
    d = _image(_side(pos, j) - pos[i], L, per)
    oi, oj, a2i, a2j, ei, ej = o[i], _side(o, j), a2[i], _side(a2, j), e[i], _side(e, j)
    wall = j < 0
    d = torch.where(wall[:, None], torch.full_like(d, 30.0), d)

    def value(n):
        return (n * d).sum(-1) - _half_width(oi, a2i, ei, n)[0] - _half_width(oj, a2j, ej, n)[0]

    n = d / d.norm(dim=-1, keepdim=True)
    g = value(n)
    for _ in range(24):
        pick = n.abs().argmin(-1, keepdim=True)
        t1 = torch.zeros_like(n).scatter_(1, pick, 1.0)
        t1 = t1 - (t1 * n).sum(-1, keepdim=True) * n
        t1 = t1 / t1.norm(dim=-1, keepdim=True)
        t2 = torch.linalg.cross(n, t1)
        g1, g2 = (t1 * d).sum(-1), (t2 * d).sum(-1)
        p11, p22, p12 = g.clone(), g.clone(), torch.zeros_like(g)
        for o_, a_, e_ in ((oi, a2i, ei), (oj, a2j, ej)):
            s, c = _half_width(o_, a_, e_, n)
            u1, u2 = (o_ * t1).sum(-1), (o_ * t2).sum(-1)
            g1, g2 = g1 - e_ * c / s * u1, g2 - e_ * c / s * u2
            p11 = p11 + a_ / s * (1 + e_ / s ** 2 * u1 * u1)
            p22 = p22 + a_ / s * (1 + e_ / s ** 2 * u2 * u2)
            p12 = p12 + a_ / s * e_ / s ** 2 * u1 * u2
        det = p11 * p22 - p12 * p12
        fine = (p11 > 0) & (det > 0)
        sc = 1.0 / (p11.abs() + p22.abs() + 1.0)
        s1 = torch.where(fine, (p22 * g1 - p12 * g2) / det, g1 * sc)
        s2 = torch.where(fine, (p11 * g2 - p12 * g1) / det, g2 * sc)
        f = (0.5 / torch.sqrt(s1 * s1 + s2 * s2).clamp_min(1e-300)).clamp_max(1.0)
        for _ in range(3):
            m = n + (f * s1)[:, None] * t1 + (f * s2)[:, None] * t2
            m = m / m.norm(dim=-1, keepdim=True)
            gm = value(m)
            f = torch.where(gm < g - 1e-13, 0.5 * f, f)
        better = gm >= g - 1e-13
        n, g = torch.where(better[:, None], m, n), torch.where(better, gm, g)
    for w, (z, s) in enumerate(dom["walls"]):
        at = j == -1 - w
        up = torch.zeros_like(n)
        up[:, 2] = 1.0
        n = torch.where(at[:, None], -float(s) * up, n)
        g = torch.where(at, s * (pos[i][:, 2] - z) - _half_width(oi, a2i, ei, up)[0], g)
    return n, g


def _surface(a, b, o, rho, n):
    """Tangent x1 along d y/dp, curvatures and cubic coefficients at rho."""
    z = (rho * o).sum(-1)
    rp = rho - z[:, None] * o
    rr = rp.norm(dim=-1)
    sp, cp = z / a, rr / b
    h = torch.sqrt(sp * sp + cp * cp)
    sp, cp = sp / h, cp / h
    pick = torch.zeros_like(o).scatter_(1, o.abs().argmin(-1, keepdim=True), 1.0)
    pole = pick - (pick * o).sum(-1, keepdim=True) * o
    pole = pole / pole.norm(dim=-1, keepdim=True)
    er = torch.where((rr > 1e-12 * b)[:, None], rp / rr.clamp_min(1e-300)[:, None], pole)
    x1 = -(b * sp)[:, None] * er + (a * cp)[:, None] * o
    x1 = x1 - (x1 * n).sum(-1, keepdim=True) * n
    x1 = x1 / x1.norm(dim=-1, keepdim=True)
    s2 = b * b * sp * sp + a * a * cp * cp
    s1 = torch.sqrt(s2)
    kk = 0.5 * (a * a - b * b) * sp * cp
    return x1, a * b / s1 ** 3, a / (b * s1), kk * a * b / s2 ** 3, kk * a / (b * s2 * s2)


def _turned(c, s, a0, a1, a2, a3):
    """A cubic's coefficients in a frame turned by (c, s) (Appendix)."""
    return (a0 * c ** 3 - a1 * s * c ** 2 + a2 * s ** 2 * c - a3 * s ** 3,
            3 * a0 * s * c ** 2 + a1 * (c ** 3 - 2 * s ** 2 * c) + a2 * (s ** 3 - 2 * s * c ** 2) + 3 * a3 * s ** 2 * c,
            3 * a0 * c * s ** 2 + a1 * (2 * c ** 2 * s - s ** 3) + a2 * (c ** 3 - 2 * c * s ** 2) - 3 * a3 * c ** 2 * s,
            a0 * s ** 3 + a1 * c * s ** 2 + a2 * c ** 2 * s + a3 * c ** 3)


def _forces(parts, i, j, n, gap, prm):
    """Pair force and torque on i and the lever arms (Sec. III B, Appendix)."""
    o, a, b, v, w = _axis(parts["q"]), parts["a"], parts["b"], parts["v"], parts["w"]
    wall = j < 0
    no = wall[:, None]

    def offset(k, m):
        a2, e = _side(b, k) ** 2, _side(a, k) ** 2 - _side(b, k) ** 2
        s, c = _half_width(_side(o, k), a2, e, m)
        return (a2 / s)[:, None] * m + (e * c / s)[:, None] * _side(o, k)

    ri, rj = offset(i, n), torch.where(no, torch.zeros_like(n), -offset(j, n))
    x1, c1, c2, G0, G2 = _surface(a[i], b[i], o[i], ri, n)
    y1, d1, d2, H0, H2 = _surface(_side(a, j), _side(b, j), _side(o, j), torch.where(no, offset(j, -n), rj), -n)
    d1, d2, H0, H2 = (torch.where(wall, torch.zeros_like(t), t) for t in (d1, d2, H0, H2))
    x2 = torch.linalg.cross(n, x1)
    cf, sf = (y1 * x1).sum(-1), (y1 * x2).sum(-1)
    r = torch.sqrt(cf * cf + sf * sf)
    cf = torch.where(wall, torch.ones_like(cf), cf / r)
    sf = torch.where(wall, torch.zeros_like(sf), sf / r)
    vj = torch.where(no, torch.zeros_like(n), _side(v, j) + torch.linalg.cross(_side(w, j), rj))
    wj = torch.where(no, torch.zeros_like(n), _side(w, j))
    dV = vj - v[i] - torch.linalg.cross(w[i], ri)
    dW = wj - w[i]
    u1, u2, u3 = ((x * dV).sum(-1) for x in (x1, x2, n))
    u4, u5, u6 = ((x * dW).sum(-1) for x in (x1, x2, n))
    A11 = 0.5 * (c1 + cf * cf * d1 + sf * sf * d2)
    A12 = 0.5 * sf * cf * (d1 - d2)
    A22 = 0.5 * (c2 + sf * sf * d1 + cf * cf * d2)
    l1 = 0.5 * (A11 + A22) + torch.sqrt((0.5 * (A11 - A22)) ** 2 + A12 ** 2)
    l2 = (A11 * A22 - A12 ** 2) / l1
    v0, v1, w0, w1 = A12, l2 - A11, l2 - A22, A12
    swap = w0 * w0 + w1 * w1 > v0 * v0 + v1 * v1
    v0, v1 = torch.where(swap, w0, v0), torch.where(swap, w1, v1)
    vn = torch.sqrt(v0 * v0 + v1 * v1)
    sx = torch.where(vn > 0, v0 / vn.clamp_min(1e-300), torch.zeros_like(vn))
    cx = torch.where(vn > 0, v1 / vn.clamp_min(1e-300), torch.ones_like(vn))
    he = torch.clamp_min(gap, prm.h_c) if prm.h_c > 0 else gap

    def log_term(delta):
        return torch.where(he < delta, torch.log1p((he - delta).clamp_max(0.0) / delta), torch.zeros_like(he))

    hn = torch.where(he < prm.delta_n, 1 / he - 1 / prm.delta_n, torch.zeros_like(he))
    lt, lr = log_term(prm.delta_t), log_term(prm.delta_r)
    sq, il = 1 / torch.sqrt(l1 * l2), 1 / (l1 + l2)
    D1, D2 = 1 / ((3 * l1 + 2 * l2) * l1), 1 / ((2 * l1 + 3 * l2) * l2)
    a1, a2, b1, b2 = c1 - l1, c1 - l2, c2 - l1, c2 - l2
    cc, ss, sc, p3 = cx * cx, sx * sx, sx * cx, 3 * PI * sq
    K11 = -PI * sq * (3 * cc * a1 * a1 * D1 + 3 * ss * a2 * a2 * D2 + 1)
    K12 = p3 * sc * (a1 * b1 * D1 - a2 * b2 * D2)
    K22 = -PI * sq * (3 * ss * b1 * b1 * D1 + 3 * cc * b2 * b2 * D2 + 1)
    K14, K15 = p3 * sc * (a1 * D1 - a2 * D2), p3 * (cc * a1 * D1 + ss * a2 * D2)
    K24, K25 = -p3 * (ss * b1 * D1 + cc * b2 * D2), p3 * sc * (b2 * D2 - b1 * D1)
    K44, K45, K55 = -p3 * (ss * D1 + cc * D2), p3 * sc * (D2 - D1), -p3 * (cc * D1 + ss * D2)
    K36 = -1.5 * PI * sq * il * sc * (c1 - c2) * (1 / l1 - 1 / l2)
    be = _turned(cf, sf, H0, torch.zeros_like(H0), H2, torch.zeros_like(H0))
    ka = _turned(cx, sx, G0 + be[0], be[1], G2 + be[2], be[3])
    r1, r2 = torch.sqrt(l1), torch.sqrt(l2)
    k0, k1, k2, k3 = ka[0] / r1 ** 3, ka[1] / (r1 * r1 * r2), ka[2] / (r1 * r2 * r2), ka[3] / r2 ** 3
    i3, i2 = 1 / (3 * l1 + 2 * l2), 1 / (2 * l1 + 3 * l2)
    Q0, Q1 = 3 * k0 * l1 + k2 * l2, k1 * l1 + 3 * k3 * l2
    Sa = (7 * l1 + 2 * l2) * k0 + (l1 + 2 * l2) * k2
    Sb = (2 * l1 + l2) * k1 + (2 * l1 + 7 * l2) * k3
    K13 = -1.5 * PI * sq * il * ((2 * r1 * Q0 - 1.5 * c1 / r1 * Sa) * cx * i3 + (2 * r2 * Q1 - 1.5 * c1 / r2 * Sb) * sx * i2
                                 + 3 * G0 * (cc / l1 + ss / l2) + G2 * (ss / l1 + cc / l2))
    K23 = -1.5 * PI * sq * il * ((-2 * r1 * Q0 + 1.5 * c2 / r1 * Sa) * sx * i3
                                 + (2 * r2 * Q1 - 1.5 * c2 / r2 * Sb) * cx * i2 + 2 * G2 * sc * (1 / l2 - 1 / l1))
    K34 = 2.25 * PI * sq * il * (Sb / r2 * i2 * cx - Sa / r1 * i3 * sx)
    K35 = -2.25 * PI * sq * il * (Sa / r1 * i3 * cx + Sb / r2 * i2 * sx)
    F1 = lt * (K11 * u1 + K12 * u2 + K14 * u4 + K15 * u5 + K13 * u3)
    F2 = lt * (K12 * u1 + K22 * u2 + K24 * u4 + K25 * u5 + K23 * u3)
    F3 = hn * p3 * il * u3 + lt * (K36 * u6 + K13 * u1 + K23 * u2 + K34 * u4 + K35 * u5)
    T4 = lt * (K14 * u1 + K24 * u2 + K34 * u3) + lr * (K44 * u4 + K45 * u5)
    T5 = lt * (K15 * u1 + K25 * u2 + K35 * u3) + lr * (K45 * u4 + K55 * u5)
    T6 = lt * K36 * u3
    F3 = prm.mu * F3
    if prm.h_c > 0:
        pen = torch.where(gap <= prm.h_c, prm.h_c - gap.clamp_min(0.0), torch.zeros_like(gap))
        F3 = F3 - prm.eps_c * pen
    F = (prm.mu * F1)[:, None] * x1 + (prm.mu * F2)[:, None] * x2 + F3[:, None] * n
    T = prm.mu * (T4[:, None] * x1 + T5[:, None] * x2 + T6[:, None] * n)
    if prm.h_c <= 0:
        dead = (gap <= 0)[:, None]
        F, T, ri, rj = (torch.where(dead, torch.zeros_like(t), t) for t in (F, T, ri, rj))
    return F, T, ri, rj


def _sums(num, i, j, F, T, ri, rj):
    f = torch.zeros(num, 3, dtype=torch.float64, device=F.device)
    t = torch.zeros_like(f)
    f.index_add_(0, i, F)
    t.index_add_(0, i, T + torch.linalg.cross(ri, F))
    at = torch.nonzero(j >= 0)[:, 0]
    f.index_add_(0, j[at], -F[at])
    t.index_add_(0, j[at], -(T + torch.linalg.cross(rj, F))[at])
    return f, t


def _exact_step(parts, dom, prm, per_pair):
    i, j = _candidates(parts, dom)
    n, gap = _closest(parts, dom, i, j)
    F, T, ri, rj = _forces(parts, i, j, n, gap, prm)
    f, t = _sums(len(parts["pos"]), i, j, F, T, ri, rj)
    out = {"force": f.T.contiguous(), "torque": t.T.contiguous(), "pair_i": None, "pair_j": None, "n": n.T.contiguous()}
    if per_pair:
        out.update(gap=gap, status=None, FT=torch.cat([F, T], 1).T.contiguous(), lever=torch.cat([ri, rj], 1).T.contiguous(),
                   iters=None)
    return out


def _subset(parts, s, e):
    return {k: v[s:e] for k, v in parts.items()}


def _exact_ensemble(case, seed):
    parts, doms, offs = _ensemble(case, seed)
    prm, got = lub.default_params(), []
    for b, dom in enumerate(doms):
        got.append(_exact_step(_subset(parts, int(offs[b]), int(offs[b + 1])), dom, prm, True))
    return {k: None if got[0][k] is None else torch.cat([d[k] for d in got], -1) for k in got[0]}


def _exact_substeps(case, seed):
    parts, dom = _suspension(case, seed)
    parts = dict(parts)
    prm = lub.default_params(h_c=0.01, eps_c=100.0)
    i, j = _candidates(parts, dom)
    a, b, dt = parts["a"], parts["b"], SUB_DT
    mass = _volume(a, b)
    ipar, iperp = 0.4 * mass * b * b, 0.2 * mass * (a * a + b * b)

    def inertia(o, x, p, q):
        c = (o * x).sum(-1, keepdim=True) * o
        return q[:, None] * (x - c) + p[:, None] * c

    for _ in range(case["sub"]):
        n, gap = _closest(parts, dom, i, j)
        f, t = _sums(len(a), i, j, *_forces(parts, i, j, n, gap, prm))
        o = _axis(parts["q"])
        parts["v"] = parts["v"] + dt * f / mass[:, None]
        parts["pos"] = parts["pos"] + dt * parts["v"]
        mom = inertia(o, parts["w"], ipar, iperp) + dt * t
        parts["q"] = _rotate(parts["q"], dt * inertia(o, mom, 1 / ipar, 1 / iperp))
        parts["w"] = inertia(_axis(parts["q"]), mom, 1 / ipar, 1 / iperp)
    out = {"force": f.T.contiguous(), "torque": t.T.contiguous(), "pair_i": None, "pair_j": None}
    for keys, key in ((("x", "y", "z"), "pos"), (("qw", "qx", "qy", "qz"), "q"), (("vx", "vy", "vz"), "v"),
                      (("wx", "wy", "wz"), "w")):
        out.update({k: parts[key][:, c].contiguous() for c, k in enumerate(keys)})
    return out


_LINKS = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
          (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


def _exact_links(case, seed):
    """Every site of i near j, every direction (Sec. II, Eq. methods:dlub)."""
    parts, dom = _suspension(case, seed)
    i, j = _candidates(parts, dom)
    pos, o, a, b = parts["pos"], _axis(parts["q"]), parts["a"], parts["b"]
    L = torch.tensor(dom["L"], dtype=torch.float64, device=pos.device)
    per = torch.tensor(dom["periodic"], device=pos.device)
    force = torch.zeros(len(i), 3, dtype=torch.float64, device=pos.device)
    torque = torch.zeros(len(i), 6, dtype=torch.float64, device=pos.device)
    mu, q_bar = lub.default_params().mu, 0.6
    ext = int(math.ceil(float(torch.maximum(a, b).max()))) + 1
    r = torch.arange(-ext, ext + 1, device=pos.device)
    grid = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)

    def quad(u, k):
        c = (o[k] * u).sum(-1)
        return (u * u).sum(-1) / b[k] ** 2 + c * c * (1 / a[k] ** 2 - 1 / b[k] ** 2)

    def hit(u, e, k):
        dc = 1 / a[k] ** 2 - 1 / b[k] ** 2
        ou, oe = (o[k] * u).sum(-1), (o[k] * e).sum(-1)
        A = 1 / b[k] ** 2 + oe * oe * dc
        B = 2 * ((u * e).sum(-1) / b[k] ** 2 + ou * oe * dc)
        C = (u * u).sum(-1) / b[k] ** 2 + ou * ou * dc - 1
        q = torch.sqrt((B * B - 4 * A * C).clamp_min(0.0))
        return (-B - q) / (2 * A), (-B + q) / (2 * A), B * B - 4 * A * C >= 0

    def curvature(u, k):
        z = (o[k] * u).sum(-1)
        s, c = z * z / a[k] ** 2, ((u * u).sum(-1) - z * z).clamp_min(0.0) / b[k] ** 2
        s1 = torch.sqrt((b[k] ** 2 * s + a[k] ** 2 * c) / (s + c))
        return 0.5 * (a[k] * b[k] / s1 ** 3 + a[k] / (b[k] * s1))

    for s in range(0, len(i), 2048):
        pi, pj = i[s:s + 2048], j[s:s + 2048]
        base = torch.floor(pos[pi])
        rj = pos[pi] + _image(_side(pos, pj) - pos[pi], L, per)
        site = (pj >= 0)[:, None] & (quad(base[:, None] + grid - pos[pi][:, None], pi[:, None]) <= 1)
        k, c = torch.nonzero(site, as_tuple=True)
        x = base[k] + grid[c]
        wide = (x - rj[k]).norm(dim=-1) <= _side(torch.maximum(a, b), pj)[k] + 3
        k, x = k[wide], x[wide]
        I, J = pi[k], pj[k].clamp_min(0)
        for vec in _LINKS:
            cr = math.sqrt(sum(v * v for v in vec))
            cv = torch.tensor(vec, dtype=torch.float64, device=pos.device)
            e = (cv / cr).expand_as(x)
            y1, y2 = x - cv, x - 2 * cv
            in1i, in1j = quad(y1 - pos[I], I) <= 1, quad(y1 - rj[k], J) <= 1
            in2i, in2j = quad(y2 - pos[I], I) <= 1, quad(y2 - rj[k], J) <= 1
            one = in1j & ~in1i
            two = ~in1j & ~in1i & in2j & ~in2i
            at = torch.nonzero(one | two)[:, 0]
            x0 = torch.where(one[at][:, None], y1[at], y2[at])
            kk, Ia, Ja, ea = k[at], I[at], J[at], e[at]
            til, _, oki = hit(x0 - pos[Ia], ea, Ia)
            _, tjh, okj = hit(x0 - rj[kk], ea, Ja)
            hs = til - tjh
            ok = oki & okj & (hs > 0) & (hs < cr)
            aI, aJ = x0 + til[:, None] * ea - pos[Ia], x0 + tjh[:, None] * ea - rj[kk]
            dv = (parts["v"][Ia] + torch.linalg.cross(parts["w"][Ia], aI)
                  - parts["v"][Ja] - torch.linalg.cross(parts["w"][Ja], aJ))
            lam = 0.5 * (curvature(aI, Ia) + curvature(aJ, Ja))
            coef = -1.5 * q_bar * mu / (cr * cr * lam) * (1 / (hs * hs) - 1 / (cr * cr)) * (ea * dv).sum(-1)
            df = torch.where(ok, coef, torch.zeros_like(coef))[:, None] * ea
            force.index_add_(0, s + kk, df)
            torque.index_add_(0, s + kk, torch.cat([torch.linalg.cross(aI, df), -torch.linalg.cross(aJ, df)], 1))
    return {"force": force.T.contiguous(), "torque": torque.T.contiguous(), "links": None}


def _exact_train(case, seed):
    x, t, w, p, m, v = (z.double() for z in _train_inputs(case, seed))
    q = p.clone().requires_grad_(True)
    at, W = 0, {}
    for key, sh in SHAPES:
        num = int(np.prod(sh))
        W[key] = q[at:at + num].view(sh)
        at += num
    h = x
    for layer in ("1", "2"):
        h = torch.nn.functional.gelu(h @ W["W" + layer].T + W["b" + layer])
    r = h @ W["W3"].T + W["b3"] - t
    r = torch.cat([(r[:, c] - (2 * PI * torch.floor(r[:, c].detach() / (2 * PI) + 0.5) if c & 1 else 0.0))[:, None]
                   for c in range(4)], 1)
    rows = 0.5 * (w * r * r).sum(1)
    rows.mean().backward()
    g = q.grad
    m = 0.9 * m + 0.1 * g
    v = 0.999 * v + 0.001 * g * g
    p = p - ADAM_LR * (m / (1 - 0.9 ** ADAM_T)) / (torch.sqrt(v / (1 - 0.999 ** ADAM_T)) + 1e-8)
    return {"grads": g, "loss": rows.detach(), "params": p, "m": m, "v": v}


def exact(case, seed):
    out = _exact(case, seed)
    if case["kind"] not in ("train", "closest"):  # zeros behind the last pair, as the arrays hold
        for key in ("n", "gap", "FT", "lever") if case["kind"] != "links" else ("force", "torque"):
            if out.get(key) is not None:
                out[key] = torch.nn.functional.pad(out[key], (0, _room(case) - out[key].shape[-1]))
    return out


def _exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "closest":
        parts, dom = _fresh_pairs(case["pairs"], seed)
        i = torch.arange(0, 2 * case["pairs"], 2, device=parts["pos"].device)
        n, gap = _closest(parts, dom, i, i + 1)
        return {"n": n.T.contiguous(), "gap": gap, "status": None}
    if kind == "ensemble":
        return _exact_ensemble(case, seed)
    if kind == "substeps":
        return _exact_substeps(case, seed)
    if kind == "links":
        return _exact_links(case, seed)
    parts, dom = _suspension(case, seed)
    if kind == "temporal":
        parts = _moved(parts, seed)
    prm = lub.default_params(precision=case.get("precision", "mixed"))
    return _exact_step(parts, dom, prm, case.get("per_pair", True))
