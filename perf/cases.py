"""The work that users of this library have it do, as cases to measure.

A luminaire here is the procedural one of plogen (a shell and a coil in the
unit cube); rays, points, targets and weights are drawn on the GPU from the
seed.  Kinds of work, by "kind":

  render   plo.render: one wavefront of rays through one plenoctree
  host     plo.render_host: the same from and to pinned host memory
  batch    Batch.render: several luminaires in one launch
  pt       plo.pt_render: a path-traced frame lit by the luminaire
  forward  Mlp.forward: the NeRF-SH network's raw outputs at points
  train    Mlp.train_step: training steps on one network
  hier     Mlp.train_step_hier: training steps on the coarse/fine pair
  distill  Mlp.distill, then a render of the tree it makes
  octopt   OctOpt.step: direct optimisation steps on an octree's leaves
"""
import math

import numpy as np
import torch

import paper_2207_05009_gb300 as plo
import plogen

PREC = {"fp32": plo.PREC_FP32, "fp16": plo.PREC_FP16, "bf16": plo.PREC_BF16}
TRANS = {"exp": plo.TRANS_EXP, "linear": plo.TRANS_LINEAR}
# leaves and nodes of the luminaire by depth, and its leaf and emissive
# segments per ray (counted for depth 10; they halve with each level)
LEAVES = {5: 4000, 6: 20656, 7: 62200, 8: 497856, 9: 3988296}
NODES = {5: 1500, 6: 6369, 7: 20929, 8: 119497, 9: 759825}
SEGMENTS = {5: 3.0, 6: 4.8, 7: 3.9, 8: 7.7, 9: 15.4}
TRUNK = 63 * 256 + 7 * 256 * 256


def listed():
    return [
        # a tile's worth of secondary rays asked of the luminaire by a host
        # renderer: the smallest call, where latency counts
        dict(name="render_d6_1k", kind="render", depth=6, degree=2, prec="fp32", trans="exp", n=1021, sigma_min=0.0,
             t_stop=0.0, aim="sphere"),
        # one bounce of a quarter-megapixel frame, 16-bit leaves, a ragged count
        dict(name="render_d8_250k_fp16", kind="render", depth=8, degree=3, prec="fp16", trans="exp", n=250007,
             sigma_min=0.0, t_stop=0.0, aim="room"),
        # a full-HD frame with the density threshold and the early stop switched on
        dict(name="render_d8_2m_bf16_stop", kind="render", depth=8, degree=3, prec="bf16", trans="exp", n=2073600,
             sigma_min=0.1, t_stop=1e-4, aim="room"),
        # a production wavefront on a deep luminaire, larger than the caches
        dict(name="render_d9_9m", kind="render", depth=9, degree=3, prec="fp32", trans="exp", n=9000001,
             sigma_min=0.0, t_stop=0.0, aim="room"),
        # a CPU renderer's emitter: rays and results in pinned host memory
        dict(name="host_d8_1m", kind="host", depth=8, degree=3, prec="fp32", trans="exp", n=1200000, sigma_min=0.0,
             t_stop=0.0, aim="room"),
        # a scene with several luminaires of different depths and degrees
        dict(name="batch_6", kind="batch", trees=6, depth=6, n=2500000, prec="fp32"),
        # a path-traced preview frame lit by the luminaire
        dict(name="pt_256", kind="pt", depth=8, degree=3, width=256, height=256, spp=4, bounces=3),
        # the network asked for its raw outputs at a ragged set of points
        dict(name="forward_200k", kind="forward", n=200001, arch="linear"),
        # training as the library's own experiment runs it
        dict(name="train_4096x128", kind="train", rays=4096, samples=128, steps=4),
        # the paper's full set-up: 1024 rays, 64 coarse + 128 fine samples
        dict(name="hier_1024", kind="hier", rays=1024, coarse=64, fine=128, steps=4),
        # the trained network turned into an octree, and a first look at it
        dict(name="distill_d7", kind="distill", depth=7, samples=8, n=65536),
        # the leaves of an octree fitted directly
        dict(name="octopt_d7", kind="octopt", depth=7, degree=2, n=32768, steps=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "render", "host", "batch", "pt", "forward", "train", "hier",
                       "distill", "octopt"])
    if kind in ("render", "host"):
        n = _log(rng, 1000, 9000000) if kind == "render" else _log(rng, 50000, 4000000)
        depth = rng.choice([6, 7, 8, 9]) if n > 200000 else rng.choice([6, 7, 8])
        return dict(kind=kind, depth=depth, degree=rng.choice([2, 3]), prec=rng.choice(["fp32", "fp32", "fp16", "bf16"]),
                    trans=rng.choice(["exp", "exp", "exp", "linear"]), n=n, sigma_min=rng.choice([0.0, 0.0, 0.1]),
                    t_stop=rng.choice([0.0, 0.0, 1e-4]), aim=rng.choice(["room", "sphere"]))
    if kind == "batch":
        return dict(kind=kind, trees=rng.randint(2, 8), depth=rng.choice([6, 7]), n=_log(rng, 100000, 4000000),
                    prec=rng.choice(["fp32", "fp16"]))
    if kind == "pt":
        return dict(kind=kind, depth=rng.choice([6, 7, 8]), degree=rng.choice([2, 3]), width=rng.randint(96, 400),
                    height=rng.randint(96, 400), spp=rng.choice([1, 2, 4]), bounces=rng.choice([1, 2, 3]))
    if kind == "forward":
        return dict(kind=kind, n=_log(rng, 5000, 500000), arch=rng.choice(["linear", "paper"]))
    if kind == "train":
        return dict(kind=kind, rays=128 * rng.randint(2, 32), samples=rng.choice([32, 64, 128]), steps=rng.randint(1, 4))
    if kind == "hier":
        return dict(kind=kind, rays=128 * rng.randint(2, 12), coarse=64, fine=rng.choice([64, 128]),
                    steps=rng.randint(1, 4))
    if kind == "distill":
        return dict(kind=kind, depth=rng.choice([5, 6, 7]), samples=rng.randint(2, 8), n=_log(rng, 4096, 65536))
    return dict(kind=kind, depth=rng.choice([6, 7]), degree=rng.choice([1, 2]), n=_log(rng, 4096, 32768),
                steps=rng.randint(4, 8))


# ---------------------------------------------------------------- inputs
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _rand(gen, *shape, dtype=torch.float32):
    return torch.rand(*shape, device="cuda", generator=gen, dtype=dtype)


def _host_tree(depth, degree, seed):
    rec = plogen.LUMINAIRE_D6 if depth <= 6 else plogen.LUMINAIRE_D10
    return plogen.luminaire_tree(rec.with_(depth=depth, sh_degree=degree, seed=20220711 + int(seed) % 1000003))


def _rays(n, aim, seed):
    """Rays aimed at uniform points of the cube, from a sphere of radius 3
    about it or from anywhere in a 10 x 10 x 3 room around it."""
    g = _gen(seed, 17)
    if aim == "sphere":
        o = torch.randn(n, 3, device="cuda", generator=g)
        o = o / o.norm(dim=1, keepdim=True) * 3.0 + 0.5
    else:
        lo = torch.tensor(plogen.ROOM_LO, device="cuda")
        hi = torch.tensor(plogen.ROOM_HI, device="cuda")
        o = lo + _rand(g, n, 3) * (hi - lo)
        inside = ((o > 0.0) & (o < 1.0)).all(dim=1)
        o[:, 0] = torch.where(inside, o[:, 0] + 1.5, o[:, 0])
    d = _rand(g, n, 3) - o
    d = d / d.norm(dim=1, keepdim=True)
    return torch.cat([o, d], 1).contiguous()


def _targets(n, seed):
    """High-dynamic-range radiances and opacities as a luminaire's images have them."""
    g = _gen(seed, 23)
    alpha = _rand(g, n).sqrt()
    rgb = alpha[:, None] * torch.exp(1.0 + 1.5 * torch.randn(n, 3, device="cuda", generator=g))
    return rgb.contiguous(), alpha.contiguous()


def _params(case):
    return plo.RenderParams(transmittance=TRANS[case["trans"]], sigma_min=case["sigma_min"], t_stop=case["t_stop"])


def _blocks(arch):
    """(rows, cols, bound factor) of the network's layers in parameter order."""
    b = [(256, 63, 1.0)] + [(256, 256, 1.0)] * 7
    return b + ([(49, 256, 0.1)] if arch == "linear" else [(1, 256, 0.1), (128, 256, 1.0), (48, 128, 0.1)])


def _weights(arch, seed, sigma_bias=0.5):
    """He-uniform weights, small biases, the output biases at a plausible density and emission level."""
    rng = np.random.default_rng([int(seed), 31])
    out = []
    for k, (rows, cols, f) in enumerate(_blocks(arch)):
        lim = f * math.sqrt(6.0 / cols)
        w = rng.uniform(-lim, lim, (rows, cols)).astype(np.float32)
        b = rng.uniform(-0.02, 0.02, rows).astype(np.float32)
        if rows in (49, 1):
            b[0] = sigma_bias
        if rows in (49, 48):
            b[(0 if rows == 48 else 1)::16] = -6.0
        out += [w.reshape(-1), b]
    return np.concatenate(out)


def _layers(flat, arch):
    """The flat parameters as (W, b) pairs in 64 bits on the GPU."""
    p = torch.from_numpy(flat).cuda().double()
    out, at = [], 0
    for rows, cols, _ in _blocks(arch):
        out.append((p[at:at + rows * cols].view(rows, cols), p[at + rows * cols:at + rows * cols + rows]))
        at += rows * cols + rows
    return out


def _encode(x):
    f = [x]
    for k in range(10):
        f += [torch.sin(math.pi * (2.0 ** k) * x), torch.cos(math.pi * (2.0 ** k) * x)]
    return torch.cat(f, 1)


def _network(layers, x, arch):
    h = _encode(x)
    for w, b in layers[:8]:
        h = torch.relu(h @ w.T + b)
    if arch == "linear":
        return h @ layers[8][0].T + layers[8][1]
    sigma = h @ layers[8][0].T + layers[8][1]
    feat = torch.relu(h @ layers[9][0].T + layers[9][1])
    return torch.cat([sigma, feat @ layers[10][0].T + layers[10][1]], 1)


L_MAX = 2000.0


def _net(case, arch, flat, salt=0, lr=5e-6):
    net = plo.Mlp(l_max=L_MAX, arch=plo.ARCH_LINEAR_HEAD if arch == "linear" else plo.ARCH_PAPER, lr0=lr, lr1=lr,
                  jitter_seed=5 + salt)
    net.set_params(flat)
    return net


def _train_batches(case, seed):
    out = []
    for k in range(case["steps"]):
        rays = _rays(case["rays"], "sphere", seed * 16 + k)
        rgb, alpha = _targets(case["rays"], seed * 16 + k)
        out.append((rays, rgb, alpha, _rand(_gen(seed * 16 + k, 29), case["rays"], case.get("samples", case.get("coarse"))),
                    _rand(_gen(seed * 16 + k, 37), case["rays"], case.get("fine", 1))))
    return out


def _batch_sizes(case, seed):
    """Uneven ray counts, one per luminaire, that sum to the case's."""
    rng = np.random.default_rng([case["trees"], case["n"], 41])
    w = np.exp(rng.uniform(0.0, 4.0, case["trees"]))
    return np.maximum(1000, (w / w.sum() * case["n"]).astype(np.int64))


def _batch_trees(case, seed):
    return [_host_tree(case["depth"] + k % 3, 2 + k % 2, seed * 16 + k) for k in range(case["trees"])]


def _batch_rays(case, seed):
    return [_rays(int(c), "room", seed * 16 + k) for k, c in enumerate(_batch_sizes(case, seed))]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("render", "host"):
        st["tree"] = plo.Tree(_host_tree(case["depth"], case["degree"], seed), PREC[case["prec"]])
        st["rays"] = _rays(case["n"], case["aim"], seed)
        st["params"] = _params(case)
        if kind == "host":
            st["rays"] = st["rays"].cpu().pin_memory()
            st["rgb"] = torch.empty(case["n"], 3).pin_memory()
            st["T"] = torch.empty(case["n"]).pin_memory()
    elif kind == "batch":
        st["trees"] = [plo.Tree(t, PREC[case["prec"]]) for t in _batch_trees(case, seed)]
        rays = _batch_rays(case, seed)
        st["batch"] = plo.Batch(st["trees"], np.concatenate([[0], np.cumsum([len(r) for r in rays])]))
        st["rays"] = torch.cat(rays)
        st["rgb"] = torch.empty(len(st["rays"]), 3, device="cuda")
        st["T"] = torch.empty(len(st["rays"]), device="cuda")
    elif kind == "pt":
        st["tree"] = plo.Tree(_host_tree(case["depth"], case["degree"], seed))
        st["seed"] = int(seed)
        st["scene"] = dict(room_min=(-1.0, -1.0, -1.0), room_max=(2.0, 2.0, 2.0), albedo=[(0.6, 0.6, 0.6)] * 6,
                           cam_pos=(0.5, 0.4, -0.9), cam_target=(0.5, 0.5, 0.5), cam_up=(0.0, 1.0, 0.0), fov_y=1.2,
                           width=case["width"], height=case["height"], max_bounces=case["bounces"],
                           emitter=plo.PT_OCTREE, box_radiance=(1.0, 1.0, 1.0))
    elif kind == "forward":
        st["net"] = _net(case, case["arch"], _weights(case["arch"], seed))
        st["points"] = _rand(_gen(seed, 43), case["n"], 3)
    elif kind == "train":
        st["net"] = _net(case, "linear", _weights("linear", seed))
        st["batches"] = _train_batches(case, seed)
    elif kind == "hier":
        st["coarse"] = _net(case, "paper", _weights("paper", seed * 2))
        st["fine"] = _net(case, "paper", _weights("paper", seed * 2 + 1), salt=1)
        st["batches"] = _train_batches(case, seed)
    elif kind == "distill":
        # the density bias at which about a quarter of the cube is kept
        flat = _weights("linear", seed, sigma_bias=0.0)
        pts = _rand(_gen(seed, 47), 8192, 3, dtype=torch.float64)
        s = torch.sort(_network(_layers(flat, "linear"), pts, "linear")[:, 0]).values
        st["net"] = _net(case, "linear", _weights("linear", seed, sigma_bias=-round(float(s[6144]), 3)))
        st["rays"] = _rays(case["n"], "sphere", seed)
    else:
        tree = _host_tree(case["depth"], case["degree"], seed)
        rng = np.random.default_rng([int(seed), 53])
        tree.sigma = rng.uniform(0.5, 2.0, tree.sigma.shape).astype(np.float32)
        tree.sh = rng.normal(0.0, 0.1, tree.sh.shape).astype(np.float32)
        tree.sh[:, :, 0] -= 18.0
        st["opt"] = plo.OctOpt(tree, L_MAX, max_rays=case["n"], lr_sigma=0.1, lr_sh=0.01, tv_sigma=1e-4, tv_sh=1e-5)
        st["batches"] = [(_rays(case["n"], "sphere", seed * 16 + k), *_targets(case["n"], seed * 16 + k))
                         for k in range(case["steps"])]
    return st


def run(state):
    kind = state["case"]["kind"]
    if kind == "render":
        rgb, T, _ = plo.render(state["tree"], state["rays"], state["params"])
        return rgb, T
    if kind == "host":
        return plo.render_host(state["tree"], state["rays"], state["params"], rgb=state["rgb"], T=state["T"])
    if kind == "batch":
        state["batch"].render(state["rays"], state["rgb"], state["T"])
        return state["rgb"], state["T"]
    if kind == "pt":
        return plo.pt_render(state["tree"], state["scene"], state["case"]["spp"], seed=state["seed"])[0]
    if kind == "forward":
        return state["net"].forward(state["points"])
    if kind == "train":
        losses = [state["net"].train_step(rays, rgb, alpha, n_samples=state["case"]["samples"], jitter=u)
                  for rays, rgb, alpha, u, _ in state["batches"]]
        return losses, state["net"].get_grads()
    if kind == "hier":
        losses = [plo.Mlp.train_step_hier(state["coarse"], state["fine"], rays, rgb, alpha,
                                          n_coarse=state["case"]["coarse"], n_fine=state["case"]["fine"], jitter=u, xi=xi)
                  for rays, rgb, alpha, u, xi in state["batches"]]
        return losses, state["coarse"].get_grads(), state["fine"].get_grads()
    if kind == "distill":
        tree = state["net"].distill(state["case"]["depth"], samples=state["case"]["samples"])
        rgb, T, _ = plo.render(tree, state["rays"], plo.RenderParams(activation=plo.ACT_SIGMOID, l_max=L_MAX))
        info = tree.info()
        return rgb, T, info["n_leaves"], info["n_nodes"]
    losses = [state["opt"].step(*b) for b in state["batches"]]
    return losses, state["opt"].read(plo.OCTOPT_GRAD_SIGMA), state["opt"].read(plo.OCTOPT_GRAD_SH)


# ---------------------------------------------------------------- what a pass cannot do without
def _render_work(n, depth, degree, prec):
    k = (degree + 1) ** 2
    rec = 12 * k if prec == "fp32" else 6 * k
    seg = SEGMENTS[depth]
    tree = 64 * NODES[depth] + 0.3 * LEAVES[depth] * rec
    seen = n * seg * (4 + 0.3 * rec)
    return 40.0 * n + min(tree, seen), n * seg * (12.0 + 0.3 * 6 * k)


def work(case):
    kind = case["kind"]
    if kind in ("render", "host"):
        b, f = _render_work(case["n"], case["depth"], case["degree"], case["prec"])
    elif kind == "batch":
        b = f = 0.0
        for k, c in enumerate(_batch_sizes(case, 0)):
            x, y = _render_work(int(c), case["depth"] + k % 3, 2 + k % 2, case["prec"])
            b, f = b + x, f + y
    elif kind == "pt":
        rays = 2 * case["bounces"] * case["spp"] * case["width"] * case["height"]
        b, f = _render_work(rays, case["depth"], case["degree"], "fp32")
        b += 12.0 * case["width"] * case["height"] - 40.0 * rays
    elif kind == "forward":
        # points in, raw outputs out, and the layer inputs that the library keeps readable
        b = case["n"] * (12.0 + 196.0 + 8 * 512.0)
        f = 2.0 * case["n"] * (TRUNK + (49 * 256 if case["arch"] == "linear" else 129 * 256 + 128 * 48))
    elif kind == "train":
        m = case["rays"] * case["samples"] * case["steps"]
        b = case["steps"] * (case["rays"] * 40.0 + 4.0 * case["rays"] * case["samples"]) + case["steps"] * 28.0 * 0.48e6
        f = 6.0 * m * (TRUNK + 49 * 256)
    elif kind == "hier":
        m = case["rays"] * (2 * case["coarse"] + case["fine"]) * case["steps"]
        b = case["steps"] * (case["rays"] * 40.0 + 4.0 * case["rays"] * (case["coarse"] + case["fine"])
                             + 2 * 28.0 * 0.51e6)
        f = 6.0 * m * (TRUNK + 129 * 256 + 128 * 48)
    elif kind == "distill":
        cells = 8.0 ** case["depth"]
        evals = cells * (1.0 + 0.25 * case["samples"])
        b, f = 0.25 * cells * 200.0 + 40.0 * case["n"], 2.0 * evals * (TRUNK + 49 * 256)
    else:
        params = LEAVES[case["depth"]] * (1 + 3 * (case["degree"] + 1) ** 2)
        seg = SEGMENTS[case["depth"]] * case["n"]
        # Adam reads and writes the parameters and both moments, writes the gradients
        b = case["steps"] * (7 * 4.0 * params + 40.0 * case["n"])
        f = case["steps"] * (14.0 * params + seg * 24.0 * (case["degree"] + 1) ** 2)
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------- the same results in 64 bits
def _sh_basis(d, degree):
    """Real orthonormal spherical harmonics, k = l (l + 1) + m, no Condon-Shortley phase."""
    x, y, z = d[:, 0], d[:, 1], d[:, 2]
    s = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    c1 = math.sqrt(3.0 / (4.0 * math.pi))
    s += [c1 * y, c1 * z, c1 * x]
    if degree >= 2:
        c2 = math.sqrt(15.0 / math.pi)
        s += [0.5 * c2 * x * y, 0.5 * c2 * y * z, 0.25 * math.sqrt(5.0 / math.pi) * (3 * z * z - 1), 0.5 * c2 * x * z,
              0.25 * c2 * (x * x - y * y)]
    if degree >= 3:
        a, b, c = math.sqrt(35.0 / (2 * math.pi)), math.sqrt(105.0 / math.pi), math.sqrt(21.0 / (2 * math.pi))
        s += [0.25 * a * y * (3 * x * x - y * y), 0.5 * b * x * y * z, 0.25 * c * y * (5 * z * z - 1),
              0.25 * math.sqrt(7.0 / math.pi) * z * (5 * z * z - 3), 0.25 * c * x * (5 * z * z - 1),
              0.25 * b * z * (x * x - y * y), 0.25 * a * x * (x * x - 3 * y * y)]
    return torch.stack(s, 1)


def _exact_render(tree, rays, trans="exp", sigma_min=0.0, t_stop=0.0):
    """March every ray cell by cell in 64 bits; the tree fills the unit cube."""
    D = tree.depth
    G = 1 << D
    child = torch.from_numpy(tree.child).cuda().long()
    sigma = torch.from_numpy(tree.sigma).cuda()
    sh = torch.from_numpy(tree.sh).cuda()
    emits = (sh != 0).flatten(1).any(1)
    n = len(rays)
    rgb = torch.zeros(n, 3, device="cuda", dtype=torch.float64)
    T_out = torch.ones(n, device="cuda", dtype=torch.float64)
    o, d = rays[:, :3].double(), rays[:, 3:].double()
    flat = d == 0.0  # such an axis never bounds the ray, unless the origin lies outside its slab
    inv = 1.0 / torch.where(flat, 1.0, d)
    ta, tb = -o * inv, (1.0 - o) * inv
    near = torch.where(flat, -math.inf, torch.minimum(ta, tb))
    t0 = near.amax(1)
    t1 = torch.where(flat, torch.where((o < 0) | (o > 1), -math.inf, math.inf), torch.maximum(ta, tb)).amin(1)
    idx = torch.nonzero((t0 < t1) & (t1 > 0)).squeeze(1)
    o, d, inv, flat, near = o[idx], d[idx], inv[idx], flat[idx], near[idx]
    t = t0[idx].clamp(min=0.0)
    up = d >= 0
    p = o + t[:, None] * d
    x = p * G
    q = torch.where((x == x.floor()) & ~up, x - 1, x.floor()).clamp(0, G - 1).long()
    at = (near == t[:, None]) & (t > 0)[:, None]  # the faces it enters by
    q = torch.where(at, torch.where(up, 0, G - 1), q)
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), tree.sh_degree)
    T = torch.ones_like(t)
    od = torch.zeros_like(t)
    C = torch.zeros(len(idx), 3, device="cuda", dtype=torch.float64)
    for _ in range(4 * G + 64):
        if not len(idx):
            break
        node = torch.zeros_like(idx)
        level = torch.zeros_like(idx)
        leaf = torch.full_like(idx, -1)
        open_ = torch.ones_like(idx, dtype=torch.bool)
        for lev in range(D):
            bits = (q >> (D - 1 - lev)) & 1
            c = child[node, bits[:, 0] | (bits[:, 1] << 1) | (bits[:, 2] << 2)]
            level = torch.where(open_, lev + 1, level)
            leaf = torch.where(open_ & (c <= -2), -c - 2, leaf)
            open_ = open_ & (c >= 0)
            node = torch.where(open_, c, node)
        down = (D - level)[:, None]
        cell = (q >> down) << down
        plane = torch.where(up, cell + (1 << down), cell)
        ts = torch.where(flat, math.inf, (plane.double() / G - o) * inv)
        te = ts.amin(1)
        out = ts <= te[:, None]
        seg = (te - t).clamp(min=0.0)
        has = leaf >= 0
        sig = torch.where(has, sigma[leaf.clamp(min=0)].double(), 0.0)
        sig = torch.where(sig < float(np.float32(sigma_min)), 0.0, sig)
        a = sig * seg
        od = od + a
        Tn = torch.exp(-od) if trans == "exp" else (1.0 - od).clamp(min=0.0)
        w = T * -torch.expm1(-a) if trans == "exp" else torch.minimum(T, a)
        hit = torch.nonzero((sig > 0) & emits[leaf.clamp(min=0)]).squeeze(1)
        for part in hit.split(1 << 20):
            e = torch.einsum("nck,nk->nc", sh[leaf[part]].double(), Y[part]).clamp(min=0.0)
            C[part] += w[part, None] * e
        T = Tn
        t = torch.maximum(te, t)
        x = ((o + t[:, None] * d) * G).floor().long()
        x = torch.minimum(torch.maximum(x, cell), cell + (1 << down) - 1)
        q = torch.where(out, torch.where(up, plane, plane - 1), x)
        done = ((q < 0) | (q >= G)).any(1) | (has & (sig > 0) & ((T < float(np.float32(t_stop))) | (T <= 0)))
        if bool(done.any()):
            rgb[idx[done]] = C[done]
            T_out[idx[done]] = T[done]
            k = ~done
            idx, o, d, inv, flat, t, up, q, Y, T, od, C = (v[k] for v in (idx, o, d, inv, flat, t, up, q, Y, T, od, C))
    return rgb, T_out


def _exact_train(case, seed):
    layers = [(w.clone().requires_grad_(), b.clone().requires_grad_()) for w, b in _layers(_weights("linear", seed), "linear")]
    flat = [p for l in layers for p in l]
    m1, m2 = [torch.zeros_like(p) for p in flat], [torch.zeros_like(p) for p in flat]
    losses = []
    N, R = case["samples"], case["rays"]
    for k, (rays, rgb, alpha, u, _) in enumerate(_train_batches(case, seed)):
        for p in flat:
            p.grad = None
        total = 0.0
        for lo in range(0, R, 512):
            r, c, al = rays[lo:lo + 512].double(), rgb[lo:lo + 512].double(), alpha[lo:lo + 512].double()
            o, d = r[:, :3], r[:, 3:]
            ta, tb = -o / d, (1.0 - o) / d
            t0 = torch.minimum(ta, tb).amax(1).clamp(min=0.0)
            t1 = torch.maximum(ta, tb).amin(1)
            j = torch.arange(N, device="cuda", dtype=torch.float64)
            t = t0[:, None] + (j + u[lo:lo + 512].double()) * ((t1 - t0) / N)[:, None]
            delta = torch.cat([t[:, 1:], t1[:, None]], 1) - t
            x = (o[:, None] + t[..., None] * d[:, None]).clamp(0.0, 1.0)
            raw = _network(layers, x.reshape(-1, 3), "linear").view(len(r), N, 49)
            a = torch.relu(raw[..., 0]) * delta
            T = torch.exp(-(torch.cumsum(a, 1) - a))
            w = T * -torch.expm1(-a)
            Y = _sh_basis(d / d.norm(dim=1, keepdim=True), 3)
            e = L_MAX * torch.sigmoid(torch.einsum("rnck,rk->rnc", raw[..., 1:].reshape(len(r), N, 3, 16), Y))
            cn = (w[..., None] * e).sum(1) / L_MAX
            res = (cn - c / L_MAX) / (cn.detach() + 0.01)
            loss = ((res ** 2).sum() + ((w.sum(1) - al) ** 2).sum()) / R
            loss.backward()
            total += float(loss.detach())
        losses.append(torch.tensor([total], dtype=torch.float64, device="cuda"))
        with torch.no_grad():
            for p, a1, a2 in zip(flat, m1, m2):
                a1.mul_(0.9).add_(0.1 * p.grad)
                a2.mul_(0.999).add_(0.001 * p.grad ** 2)
                p -= 5e-6 * (a1 / (1 - 0.9 ** (k + 1))) / (torch.sqrt(a2 / (1 - 0.999 ** (k + 1))) + 1e-8)
    return losses, torch.cat([p.grad.reshape(-1) for p in flat]).cpu().numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("render", "host"):
        rgb, T = _exact_render(_host_tree(case["depth"], case["degree"], seed), _rays(case["n"], case["aim"], seed),
                               case["trans"], case["sigma_min"], case["t_stop"])
        return (rgb, T) if kind == "render" else (rgb.cpu(), T.cpu())
    if kind == "batch":
        got = [_exact_render(t, r) for t, r in zip(_batch_trees(case, seed), _batch_rays(case, seed))]
        return torch.cat([g[0] for g in got]), torch.cat([g[1] for g in got])
    if kind == "forward":
        layers = _layers(_weights(case["arch"], seed), case["arch"])
        pts = _rand(_gen(seed, 43), case["n"], 3).double()
        return torch.cat([_network(layers, x, case["arch"]) for x in pts.split(65536)])
    if kind == "train":
        return _exact_train(case, seed)
    # a frame's paths and an octree's kept cells branch on computed numbers; the
    # pair's fine samples follow the coarse network's weights; the leaves' steps
    # follow the sign of small gradients
    return None
