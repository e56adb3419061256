"""What the framework is measured on: the calls its users make, over their real range of sizes.

A case is a dict of plain values.  Kinds:

* ``chains``  advance a chain set and resolve its image: Jump Restore (uniform or learned regeneration, with or
  without completing the open tours), the MH baseline, and the Langevin (MALA) local moves;
* ``batch``   many chain sets of uneven size advanced together, replayed from a CUDA graph;
* ``density`` / ``sample``  rows through the regeneration flow, both directions;
* ``train``   Adam steps of the flow on a replay ring of chain states;
* ``render``  plain path tracing, which makes the converged references.

The scenes are the package's seeded ones; geometry arrays are built once per process and uploaded anew (with a new
BVH) in every ``prepare``.
"""
import functools
import math

import numpy as np
import torch

from paper_2409_07148_gb300 import jr, scenes
from paper_2409_07148_gb300.flowinit import init_flow_params

LAYERS, HIDDEN, BINS, PAD, FLOOR = 6, 64, 16, 16, 1e-3  # the flow's documented layout


def listed():
    return [
        # the smallest render: the 24-triangle box, a few hundred chains for many steps (latency of one step)
        dict(name="box_256_chains", kind="chains", scene="cornell", width=64, height=64, depth=3, chains=256, steps=400,
             flow_dim=0, beta=0.0, tours=False, mode="restore", rao=False),
        # a preview: an odd number of chains, too few for the wavefront, on a 40k-triangle scene and an oblong image
        dict(name="spheres_10007_chains", kind="chains", scene="cornell_spheres", width=200, height=136, depth=8,
             chains=10007, steps=32, flow_dim=0, beta=0.0, tours=False, mode="restore", rao=False),
        # the benchmark's workload: 40k triangles, 512 x 512, depth 8, 2^20 chains
        dict(name="spheres_1m_chains", kind="chains", scene="cornell_spheres", width=512, height=512, depth=8,
             chains=1 << 20, steps=16, flow_dim=0, beta=0.0, tours=False, mode="restore", rao=False),
        # a checkpoint of the completed-tour estimator on the caustic: advance, finish every open tour, resolve
        dict(name="caustic_tours", kind="chains", scene="caustic_slit", width=512, height=512, depth=10,
             chains=1 << 18, steps=16, flow_dim=0, beta=0.0, tours=True, mode="restore", rao=False),
        # learned regeneration: a flow over the leading 8 of 22 coordinates inside the chains
        dict(name="caustic_learned", kind="chains", scene="caustic_slit", width=512, height=512, depth=10,
             chains=1 << 18, steps=8, flow_dim=8, beta=0.15, tours=False, mode="restore", rao=False),
        # the largest scene: 2M triangles, 256 emitters, 2048 x 2048, depth 12
        dict(name="terrain_1m_chains", kind="chains", scene="terrain", width=2048, height=2048, depth=12,
             chains=1 << 20, steps=4, flow_dim=0, beta=0.0, tours=False, mode="restore", rao=False),
        # Langevin local moves: the path contribution's gradient in every step
        dict(name="spheres_mala", kind="chains", scene="cornell_spheres", width=256, height=256, depth=8,
             chains=1 << 15, steps=8, flow_dim=0, beta=0.0, tours=False, mode="mala", rao=False),
        # eight interiors of 1k-200k triangles and uneven image sizes in one batch, one chain per pixel
        dict(name="batch_8_rooms", kind="batch", sets=8, geometry=0, steps=4, block=0),
        # density rows of the full-dimensional flow (the candidates that become lit states of 2^18 chains)
        dict(name="flow_density_22", kind="density", dim=22, rows=1 << 18),
        # sampling rows of the leading-coordinate flow: the flow draws of a step, a ragged count
        dict(name="flow_sample_8", kind="sample", dim=8, rows=40003),
        # one epoch's training: 25 Adam steps of 8192 rows on a ring of 2^18 states
        dict(name="flow_train_22", kind="train", dim=22, batch=8192, iters=25, ring=1 << 18, lr=3e-3),
        # a share of a converged reference
        dict(name="spheres_reference", kind="render", scene="cornell_spheres", width=512, height=512, depth=8,
             samples=1 << 21),
    ]


def _spread(rng, lo, hi):
    """An integer log-uniform in [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["chains", "chains", "chains", "learned", "batch", "density", "sample", "train", "render"])
    if kind == "density" or kind == "sample":
        return dict(kind=kind, dim=2 * rng.randint(2, 13), rows=_spread(rng, 1000, 1 << 18))
    if kind == "train":
        return dict(kind=kind, dim=2 * rng.randint(3, 13), batch=64 * _spread(rng, 8, 128), iters=rng.randint(4, 25),
                    ring=_spread(rng, 1 << 14, 1 << 18), lr=3e-3)
    if kind == "batch":
        return dict(kind=kind, sets=rng.randint(2, 8), geometry=rng.randint(1, 5), steps=rng.randint(1, 4),
                    block=rng.choice([0, 0, 64, 128]))
    if kind == "learned":
        return dict(kind="chains", scene="caustic_slit", width=_spread(rng, 100, 512), height=_spread(rng, 100, 512),
                    depth=rng.randint(4, 10), chains=_spread(rng, 3000, 1 << 18), steps=rng.randint(1, 8),
                    flow_dim=2 * rng.randint(2, 5), beta=round(rng.uniform(0.05, 0.3), 3), tours=rng.random() < 0.3,
                    mode="restore", rao=False)
    scene = rng.choice(["cornell", "cornell_spheres", "cornell_spheres", "caustic_slit", "terrain"])
    depth = {"cornell": rng.randint(2, 6), "cornell_spheres": rng.randint(3, 8), "caustic_slit": rng.randint(5, 10),
             "terrain": rng.randint(4, 12)}[scene]
    width, height = _spread(rng, 64, 800), _spread(rng, 64, 800)
    if kind == "render":
        return dict(kind=kind, scene=scene, width=width, height=height, depth=depth,
                    samples=_spread(rng, 50000, 1 << 21))
    mode = rng.choice(["restore", "restore", "restore", "mh", "mala"])
    if mode == "mala":
        chains, steps = _spread(rng, 500, 1 << 15), rng.randint(1, 8)
    else:
        chains = _spread(rng, 200, 1 << 20)
        steps = max(1, min(200, int((1 << 22) // chains)))
        if scene == "terrain":
            steps = min(steps, 4)
    return dict(kind="chains", scene=scene, width=width, height=height, depth=depth, chains=chains, steps=steps,
                flow_dim=0, beta=0.0, tours=mode == "restore" and rng.random() < 0.2, mode=mode,
                rao=mode == "restore" and rng.random() < 0.3)


# ---------------------------------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _geometry(name, width, height, depth):
    return getattr(scenes, name)(width=width, height=height, depth=depth)


@functools.lru_cache(maxsize=None)
def _rooms(geometry, sets):
    return scenes.batched_workload(seed=geometry, n_scenes=sets)


def _flow_params(dim, seed):
    """A flow with structure: the package's initial hidden layers, and output layers that make logits of order 1."""
    perm, w = init_flow_params(dim, seed)
    rng = np.random.default_rng(seed + 1)
    n = dim // 2 * BINS
    at = w.shape[1] - n * (HIDDEN + 1)
    w[:, at:] = rng.normal(0.0, 0.15, (LAYERS, n * (HIDDEN + 1)))
    return perm, w


def _states(dim, n, seed):
    """Rows like chain states: a uniform background and a concentrated part (film and first bounces), in [0, 1)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((dim, n), generator=g, device="cuda")
    part = torch.rand(n, generator=g, device="cuda") < 0.6
    spread = 0.08 * torch.randn((dim, n), generator=g, device="cuda")
    centre = torch.rand((dim, 1), generator=g, device="cuda")
    x = torch.where(part[None, :], (centre + spread).remainder(1.0), x)
    x = x.clamp_(0.0, 1.0 - 2.0 ** -24).contiguous()
    w = torch.rand(n, generator=g, device="cuda") * 0.9 + 0.05
    return x, w


class _State:
    pass


def _image(sc):
    return torch.empty((sc.height, sc.width, 3), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    s = _State()
    s.case = case
    kind = case["kind"]
    if kind == "chains":
        sc = _geometry(case["scene"], case["width"], case["height"], case["depth"])
        s.scene = jr.Scene(sc)
        flags = {"restore": 0, "mh": jr.JR_FLAG_MH, "mala": jr.JR_FLAG_MALA}[case["mode"]]
        if case["rao"]:
            flags |= jr.JR_FLAG_RAO_BLACKWELL
        s.chains = jr.Chains(s.scene, sc.width, sc.height, sc.depth, case["chains"], seed=seed, flags=flags,
                             sigma=0.02 if case["mode"] == "mala" else 0.01, burn_in=0)
        s.image = _image(sc)
        if case["flow_dim"]:
            s.flow = jr.Flow(case["flow_dim"], *_flow_params(case["flow_dim"], seed))
            jr.set_flow(s.chains, s.flow, case["beta"])
    elif kind == "batch":
        rooms = _rooms(case["geometry"], case["sets"])
        s.sets = [jr.Chains(jr.Scene(sc), sc.width, sc.height, sc.depth, sc.width * sc.height, seed=seed + 7919 * k)
                  for k, sc in enumerate(rooms)]
        s.batch = jr.Batch(s.sets)
        s.batch.set_block(case["block"])
        s.images = [_image(sc) for sc in rooms]
    elif kind in ("density", "sample"):
        s.flow = jr.Flow(case["dim"], *_flow_params(case["dim"], seed))
        s.x = _states(case["dim"], case["rows"], seed)[0]
    elif kind == "train":
        s.flow = jr.Flow(case["dim"], *_flow_params(case["dim"], seed))
        s.ring = jr.ReplayBuffer(case["dim"], case["ring"])
        s.ring.x, s.ring.w = _states(case["dim"], case["ring"], seed)
        s.ring.total.fill_(case["ring"])
        s.seed = seed
    else:
        sc = _geometry(case["scene"], case["width"], case["height"], case["depth"])
        s.scene = jr.Scene(sc)
        s.seed = seed
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "chains":
        s.chains.advance(case["steps"])
        out = {}
        if case["tours"]:
            out["open_tours"] = jr.complete_tours(s.chains)
        out["image"] = s.chains.resolve(out=s.image)
        out["x"], out["w"] = jr.snapshot(s.chains)
        return out
    if kind == "batch":
        s.batch.advance_graph(case["steps"])
        return {"images": [c.resolve(out=im) for c, im in zip(s.sets, s.images)],
                "states": [jr.snapshot(c) for c in s.sets]}
    if kind == "density":
        return s.flow.log_density(s.x)
    if kind == "sample":
        z = s.x.clone()
        return {"log_q": s.flow.sample(z), "x": z}
    if kind == "train":
        losses = s.flow.train_replay(s.ring, case["iters"], batch=case["batch"], lr=case["lr"], seed=s.seed)
        return {"losses": losses, "params": s.flow.get_params()}
    return jr.render_pt(s.scene, case["width"], case["height"], case["depth"], case["samples"], seed=s.seed)


# ------------------------------------------------------------------------------------------------------------ work
# Per path: rays cast and arithmetic per ray (slab tests of the nodes a ray enters, triangle tests, one shading),
# counted on these scenes.
_RAYS = {"cornell": (0.9, 150.0), "cornell_spheres": (0.52, 570.0), "caustic_slit": (0.16, 420.0),
         "terrain": (0.18, 900.0), "rooms": (0.95, 750.0)}


def _path_flops(scene, depth):
    share, per_ray = _RAYS[scene]
    return max(1.0, share * (depth + 1)) * per_ray


def _flow_flops(dim):
    a = dim // 2
    return LAYERS * (2.0 * HIDDEN * (a + HIDDEN + a * BINS) + 6.0 * a * BINS)


def _chain_work(scene, width, height, depth, chains, steps):
    dim = 2 + 2 * depth
    # the state read, the state and its weight written, the image written; the scene stays in the caches
    return 4.0 * chains * (2 * dim + 1) + 12.0 * width * height, 1.0 * chains * steps * _path_flops(scene, depth)


def work(case):
    kind = case["kind"]
    if kind == "chains":
        b, f = _chain_work(case["scene"], case["width"], case["height"], case["depth"], case["chains"], case["steps"])
        if case["flow_dim"]:
            f += case["chains"] * case["steps"] * case["beta"] * _flow_flops(case["flow_dim"])
        return {"bytes": b, "flops": f}
    if kind == "batch":
        b = f = 0.0
        for sc in _rooms(case["geometry"], case["sets"]):
            bb, ff = _chain_work("rooms", sc.width, sc.height, sc.depth, sc.width * sc.height, case["steps"])
            b, f = b + bb, f + ff
        return {"bytes": b, "flops": f}
    if kind == "density":
        return {"bytes": 4.0 * case["rows"] * (case["dim"] + 1), "flops": case["rows"] * _flow_flops(case["dim"])}
    if kind == "sample":
        return {"bytes": 4.0 * case["rows"] * (2 * case["dim"] + 1), "flops": case["rows"] * _flow_flops(case["dim"])}
    if kind == "train":
        a = case["dim"] // 2
        params = LAYERS * (HIDDEN * (PAD + HIDDEN + 2) + a * BINS * (HIDDEN + 1))
        return {"bytes": 4.0 * case["iters"] * case["batch"] * (case["dim"] + 1) + 4.0 * 6 * params * case["iters"],
                "flops": 3.0 * case["iters"] * case["batch"] * _flow_flops(case["dim"])}
    return {"bytes": 32.0 * case["width"] * case["height"],
            "flops": case["samples"] * _path_flops(case["scene"], case["depth"])}


# ----------------------------------------------------------------------------------------------------------- exact
def _layer64(perm, w, dim, l):
    a, n = dim // 2, dim // 2 * BINS
    sizes = [HIDDEN * PAD, HIDDEN, HIDDEN * HIDDEN, HIDDEN, n * HIDDEN, n]
    w1, b1, w2, b2, w3, b3 = torch.split(w[l], sizes)
    p = torch.as_tensor(perm[l], dtype=torch.long, device="cuda")
    return p[:a], p[a:], (w1.view(HIDDEN, PAD)[:, :a], b1, w2.view(HIDDEN, HIDDEN), b2, w3.view(n, HIDDEN), b3)


def _masses64(x, net):
    """Bin masses [n, a, BINS] of the transformed coordinates from the conditioning ones, x [n, a]."""
    w1, b1, w2, b2, w3, b3 = net
    h = torch.relu(x @ w1.T + b1)
    h = torch.relu(h @ w2.T + b2)
    o = (h @ w3.T + b3).view(x.shape[0], -1, BINS)
    return (1.0 - FLOOR) * torch.softmax(o, -1) + FLOOR / BINS


def _density64(perm, w, dim, x):
    """log q of rows x [n, dim]."""
    cols = list(x.unbind(1))
    lq = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for l in range(LAYERS):
        keep, move, net = _layer64(perm, w, dim, l)
        keep, move = keep.tolist(), move.tolist()
        q = _masses64(torch.stack([cols[c] for c in keep], 1), net)
        t = torch.stack([cols[c] for c in move], 1)
        b = (t.detach() * BINS).long().clamp(0, BINS - 1)
        qb = q.gather(-1, b[..., None])[..., 0]
        lo = (q * (torch.arange(BINS, device="cuda") < b[..., None])).sum(-1)
        t = lo + (t * BINS - b) * qb
        lq = lq + torch.log(BINS * qb).sum(1)
        for j, c in enumerate(move):
            cols[c] = t[:, j]
    return lq


def _sample64(perm, w, dim, x):
    x = x.clone()
    lq = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for l in reversed(range(LAYERS)):
        keep, move, net = _layer64(perm, w, dim, l)
        q = _masses64(x[:, keep], net)
        v = x[:, move]
        cum = torch.cumsum(q, -1)
        b = (cum <= v[..., None]).sum(-1).clamp(max=BINS - 1)
        qb = q.gather(-1, b[..., None])[..., 0]
        lo = cum.gather(-1, b[..., None])[..., 0] - qb
        x[:, move] = ((b + (v - lo) / qb) / BINS).clamp(0.0, 1.0 - 2.0 ** -24)
        lq += torch.log(BINS * qb).sum(1)
    return x, lq


def _train64(case, seed):
    dim, n, batch = case["dim"], case["ring"], min(case["batch"], case["ring"] // 64 * 64)
    perm, w0 = _flow_params(dim, seed)
    x, wt = _states(dim, n, seed)
    x, wt = x.T.double(), wt.double()
    w = torch.as_tensor(w0, device="cuda").double().requires_grad_(True)
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    mask, losses = (1 << 64) - 1, []
    rng = (seed * 0x9E3779B97F4A7C15 + 0xD1B54A32D192ED03) & mask
    for it in range(case["iters"]):
        # the minibatch window of this step (splitmix64)
        rng ^= rng >> 30
        rng = (rng * 0xBF58476D1CE4E5B9) & mask
        rng ^= rng >> 27
        rng = (rng * 0x94D049BB133111EB) & mask
        rng ^= rng >> 31
        off = rng % (n - batch + 1)
        ww = wt[off:off + batch]
        loss = -(ww * _density64(perm, w, dim, x[off:off + batch])).sum() / ww.sum()
        (g,) = torch.autograd.grad(loss, w)
        losses.append(loss.detach())
        with torch.no_grad():
            m.mul_(0.9).add_(g, alpha=0.1)
            v.mul_(0.999).addcmul_(g, g, value=0.001)
            t = it + 1
            w -= case["lr"] * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"losses": torch.stack(losses), "params": w.detach().reshape(-1)}


def exact(case, seed):
    """The flow's results in 64 bits.  Chains have none: an image is a sum over random paths, and their states follow
    decisions that the arithmetic itself makes."""
    kind = case["kind"]
    if kind == "train":
        return _train64(case, seed)
    if kind not in ("density", "sample"):
        return None
    perm, w = _flow_params(case["dim"], seed)
    w = torch.as_tensor(w, device="cuda").double()
    x = _states(case["dim"], case["rows"], seed)[0].T.double()
    if kind == "density":
        return _density64(perm, w, case["dim"], x)
    y, lq = _sample64(perm, w, case["dim"], x)
    return {"log_q": lq, "x": y.T.contiguous()}
