"""The work that a user of the library has it do, as cases that can be timed and compared.

A case names an operation ("op"), its kernel, the numbers of sources and queries and the options of
the call. Inputs are drawn on the GPU from the seed alone: surface samples of unions of random
ellipsoids and boxes with area weights and outward normals, rescaled into [-1, 1]^3 (uniform points
of the unit cube for the small problem), queried on grids, on shuffled slice planes or at random.

The operations, each through the public entry points:
  step         sbh_build and sbh_eval: a new point set and one evaluation of it
  host         sbh_solve_host: the same from page-locked host buffers, results back on the host
  multi        sbh_multi_plan_launch: many prebuilt problems of very different sizes in one launch
  grad         StochasticSum and its backward pass: estimate and query gradient
  learned      sbh_eval_learned: the estimate with the learned child proposal
  train        sbh_mlp_create and sbh_mlp_train: fit the proposal to a tree
  bh           sbh_eval_bh on a prebuilt tree: deterministic Barnes-Hut
  bh_step      sbh_build and sbh_eval_bh: a new point set, its 8-ary tree and one evaluation
  brute        sbh_eval_brute with FP64 accumulation: the exact sum, the reference of every error
  brute_grad   sbh_eval_brute_grad: the exact sum and its query gradient
"""
import math

import numpy as np
import torch

import paper_2506_02219_gb300 as sbh

SOFTENING = 1e-3
ALPHA = 200.0


def listed():
    return [
        # a small interactive problem: 4,096 masses and a 64 x 64 plane of queries, where the latency
        # of the build's many steps is what a user waits for
        {"name": "step_cube", "op": "step", "kernel": "coulomb", "shape": "cube", "n": 4096, "queries": "plane",
         "nq": 64 * 64, "S": 1, "leaf": 1},
        # the headline configuration: winding numbers of 2^20 oriented samples on a 256^3 grid
        {"name": "step_winding", "op": "step", "kernel": "winding", "shape": "union", "n": 1 << 20, "queries": "grid",
         "nq": 1 << 24, "S": 1, "leaf": 1},
        # smooth distances on a shuffled 1000 x 1000 slice plane through 2^22 samples: a large source
        # set, evaluated once, so that the build weighs as much as the evaluation
        {"name": "step_slice_smooth", "op": "step", "kernel": "smoothdist", "shape": "union", "n": 1 << 22,
         "queries": "plane", "nq": 1000 * 1000, "S": 1, "leaf": 1},
        # a potential at an odd number of points in and around the sources, from host memory to host memory
        {"name": "host_coulomb", "op": "host", "kernel": "coulomb", "shape": "union", "n": 300007, "queries": "around",
         "nq": 1000003, "S": 1, "leaf": 1},
        # 64 independent sets, sources log-uniform in 2^10 .. 2^20 and queries in 2^8 .. 2^18, in one launch
        {"name": "multi_smooth", "op": "multi", "kernel": "smoothdist", "shape": "cube", "sets": 64, "n": 1 << 20,
         "queries": "around", "nq": 1 << 18, "S": 2, "leaf": 2},
        # forward and backward through the estimate, as in an optimisation over query positions
        {"name": "grad_winding", "op": "grad", "kernel": "winding", "shape": "union", "n": 1 << 20,
         "queries": "random", "nq": 1500007, "S": 1, "leaf": 1},
        # the learned child proposal on the slice plane
        {"name": "learned_slice", "op": "learned", "kernel": "coulomb", "shape": "union", "n": 1 << 20,
         "queries": "plane", "nq": 1000 * 1000, "S": 1, "leaf": 1, "near": 0.25},
        # fitting that proposal: 256 training queries, 20 full-batch steps
        {"name": "train_winding", "op": "train", "kernel": "winding", "shape": "union", "n": 1 << 17,
         "queries": "random", "nq": 256, "leaf": 1, "near": 0.5, "steps": 20},
        # Barnes-Hut with warp voting on a 128^3 grid, neighbouring queries side by side
        {"name": "bh_grid", "op": "bh", "kernel": "winding", "shape": "union", "n": 1 << 20, "queries": "grid",
         "nq": 1 << 21, "leaf": 1, "theta": 0.5, "vote": True},
        # a new point set and Barnes-Hut at random points in no order, every query for itself
        {"name": "bh_step_random", "op": "bh_step", "kernel": "coulomb", "shape": "union", "n": 1 << 18,
         "queries": "random", "nq": 1000 * 1000, "leaf": 4, "theta": 0.8, "vote": False},
        # the error reference of the benchmark: 65,536 queries against every one of 2^20 sources
        {"name": "brute_winding", "op": "brute", "kernel": "winding", "shape": "union", "n": 1 << 20,
         "queries": "random", "nq": 1 << 16},
        # the reference of the gradients' errors, with a few thousand queries
        {"name": "brute_grad_smooth", "op": "brute_grad", "kernel": "smoothdist", "shape": "cube", "n": 1 << 19,
         "queries": "random", "nq": 5001},
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "host", "multi", "grad", "learned", "train", "bh", "bh_step", "brute",
                     "brute_grad"])
    kernel = rng.choice(["coulomb", "winding", "smoothdist"])
    c = {"op": op, "kernel": kernel, "shape": "union" if kernel == "winding" else rng.choice(["cube", "union"])}
    where = rng.choice(["plane", "grid", "random", "around"])
    leaf = rng.choice([1, 1, 1, 2, 4, 7])
    if op == "step":
        return {**c, "n": _log(rng, 1000, 1 << 22), "queries": where, "nq": _log(rng, 1000, 1 << 22),
                "S": rng.choice([1, 1, 2, 3]), "leaf": leaf}
    if op == "host":
        return {**c, "n": _log(rng, 4096, 1 << 20), "queries": where, "nq": _log(rng, 4096, 1 << 21),
                "S": rng.choice([1, 2]), "leaf": leaf}
    if op == "multi":
        return {**c, "shape": "cube", "sets": rng.randint(5, 64), "n": _log(rng, 1 << 12, 1 << 20), "queries": "around",
                "nq": _log(rng, 1 << 9, 1 << 18), "S": rng.choice([1, 2]), "leaf": leaf}
    if op == "grad":
        return {**c, "n": _log(rng, 4096, 1 << 20), "queries": where, "nq": _log(rng, 1000, 1 << 21),
                "S": rng.choice([1, 2]), "leaf": leaf}
    if op == "learned":
        return {**c, "n": _log(rng, 4096, 1 << 20), "queries": where, "nq": _log(rng, 1000, 1 << 20), "S": 1,
                "leaf": leaf, "near": rng.choice([0.25, 0.5])}
    if op == "train":
        return {**c, "n": _log(rng, 4096, 1 << 17), "queries": "random", "nq": _log(rng, 32, 256), "leaf": leaf,
                "near": rng.choice([0.25, 0.5]), "steps": rng.randint(5, 20)}
    if op in ("bh", "bh_step"):
        theta = rng.choice([0.5, 0.8, 1.0])
        vote = rng.random() < 0.5
        most = 1 << 17 if vote and where == "random" else 1 << 20
        return {**c, "n": _log(rng, 4096, 1 << 20), "queries": where, "nq": _log(rng, 1000, most), "leaf": leaf,
                "theta": theta, "vote": vote}
    n = _log(rng, 1 << 13, 1 << 20)
    most = min(1 << 16, (1 << 36) // n) if op == "brute" else min(1 << 14, (1 << 33) // n)
    return {**c, "n": n, "queries": "random", "nq": _log(rng, 500, most)}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _rotation(g):
    w, x, y, z = (g / g.norm()).tolist()
    return torch.tensor([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                         [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                         [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])


def _union(n, seed):
    """n area-uniform samples on the outside of a union of 8 random ellipsoids and 4 boxes, in random
    order, rescaled into [-1, 1]^3: points, area weights (a shape's area over the samples drawn on it),
    outward normals."""
    cpu = torch.Generator().manual_seed(seed)
    gpu = torch.Generator(device="cuda").manual_seed(seed)
    shapes = []
    for k in range(12):
        c = torch.rand(3, generator=cpu) * 1.2 - 0.6
        if k < 8:
            ax = torch.rand(3, generator=cpu) * 0.35 + 0.15
            shapes.append((True, c.cuda(), ax.cuda(), _rotation(torch.randn(4, generator=cpu)).cuda()))
        else:
            shapes.append((False, c.cuda(), (torch.rand(3, generator=cpu) * 0.3 + 0.1).cuda(), torch.eye(3).cuda()))

    def inside(s, p):
        x = (p - s[1]) @ s[3]
        return ((x / s[2]) ** 2).sum(1) < 1 if s[0] else ((x.abs() < s[2]).all(1))

    areas = []
    for ball, _, h, _ in shapes:
        a, b, c = h.tolist()
        q = 1.6075  # Thomsen's formula for an ellipsoid's area (within 1%)
        areas.append(4 * math.pi * (((a * b) ** q + (a * c) ** q + (b * c) ** q) / 3) ** (1 / q) if ball
                     else 8 * (a * b + b * c + a * c))
    P, N, own, have, drawn = [], [], [], 0, torch.zeros(12, device="cuda")
    while have < n:
        for i, s in enumerate(shapes):
            m = int(math.ceil(2.2 * n * areas[i] / sum(areas))) + 64
            if s[0]:
                u = torch.randn(m, 3, generator=gpu, device="cuda")
                u = u / u.norm(dim=1, keepdim=True)
                stretch = (u / s[2]).norm(dim=1)  # area element of the map of the sphere onto the ellipsoid
                u = u[torch.rand(m, generator=gpu, device="cuda") < stretch / (1 / s[2]).max()]
                p, v = u * s[2], u / s[2]
                v = v / v.norm(dim=1, keepdim=True)
            else:
                m = m // 2
                face = s[2].new_tensor([s[2][1] * s[2][2], s[2][0] * s[2][2], s[2][0] * s[2][1]])
                ax = torch.multinomial(face, m, replacement=True, generator=gpu)
                sign = (torch.rand(m, generator=gpu, device="cuda") < 0.5).float() * 2 - 1
                p = torch.rand(m, 3, generator=gpu, device="cuda") * 2 - 1
                p.scatter_(1, ax[:, None], sign[:, None])
                v = torch.zeros_like(p).scatter_(1, ax[:, None], sign[:, None])
                p = p * s[2]
            p = p @ s[3].T + s[1]
            drawn[i] += p.shape[0]
            out = torch.ones(p.shape[0], dtype=torch.bool, device="cuda")
            for j, o in enumerate(shapes):
                if j != i:
                    out &= ~inside(o, p)
            P.append(p[out])
            N.append((v @ s[3].T)[out])
            own.append(torch.full((P[-1].shape[0],), i, device="cuda"))
            have += P[-1].shape[0]
    P, N, own = torch.cat(P), torch.cat(N), torch.cat(own)
    at = torch.randperm(have, generator=gpu, device="cuda")[:n]
    P, N = P[at], N[at]
    w = (torch.tensor(areas, device="cuda") / drawn)[own[at]] * (have / n)
    lo, hi = P.amin(0), P.amax(0)
    scale = float(2 / (hi - lo).max() * 0.999)
    return ((P - (lo + hi) / 2) * scale).contiguous(), w * (scale * scale), N.contiguous()


def _sources(case, n, seed):
    if case["shape"] == "union":
        p, w, v = _union(n, seed)
        return p, (torch.ones_like(w) if case["kernel"] == "smoothdist" else w), (v if case["kernel"] == "winding" else None)
    gpu = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.rand(n, 3, generator=gpu, device="cuda")
    w = torch.rand(n, generator=gpu, device="cuda") + 0.5
    v = None
    if case["kernel"] == "winding":
        v = torch.randn(n, 3, generator=gpu, device="cuda")
        v = (v / v.norm(dim=1, keepdim=True)).contiguous()
    return p, (torch.ones_like(w) if case["kernel"] == "smoothdist" else w), v


def _queries(case, p, nq, seed):
    """nq queries in the sources' bounding box: a slice plane in random order, a grid (x fastest),
    uniform points in no order, or uniform points of the box grown by half on each side."""
    gpu = torch.Generator(device="cuda").manual_seed(seed + 1)
    lo, hi = p.amin(0), p.amax(0)
    if case["queries"] in ("random", "around"):
        q = torch.rand(nq, 3, generator=gpu, device="cuda")
        q = q if case["queries"] == "random" else q * 2 - 0.5
        return (lo + q * (hi - lo)).contiguous()
    d = 2 if case["queries"] == "plane" else 3
    r = int(math.ceil(round(nq ** (1.0 / d), 6)))
    k = torch.arange(nq, device="cuda")
    if d == 2:
        k = torch.randperm(r * r, generator=gpu, device="cuda")[:nq]
    shift = float(torch.rand(1, generator=gpu, device="cuda"))  # the grid's offset: half a cell on average
    x = torch.stack([k % r, (k // r) % r, k // (r * r)], 1).float()
    x = (x + shift) / r
    if d == 2:
        x[:, 2] = 0.35 + 0.3 * shift
    return (lo + x * (hi - lo)).contiguous()


def _proposal(seed):
    """Weights of a child proposal: random ones, and on them the two habits of a trained proposal, to
    prefer children near the query and heavy ones."""
    rng = np.random.default_rng(seed)
    w1, w2 = rng.normal(0, 0.15, (32, 6)), rng.normal(0, 0.05, (32, 32))
    w3 = rng.normal(0, 0.15, 32)
    w1[:4], w2[:4], w3[:4] = 0.0, 0.0, (-1.5, 1.5, 0.7, -0.7)
    w1[0, 0], w1[1, 0], w1[2, 1], w1[3, 1] = 1.0, -1.0, 1.0, -1.0
    w2[range(4), range(4)] = 1.0
    return np.concatenate([w1.ravel(), np.zeros(32), w2.ravel(), np.zeros(32), w3, [0.0]]).astype(np.float32)


def prepare(case, seed):
    op = case["op"]
    st = {"case": case, "seed": seed, "kw": {"softening": SOFTENING, "alpha": ALPHA}}
    if op == "multi":
        rng = np.random.default_rng(case["sets"])  # the sizes belong to the case, the points to the seed
        st["trees"], st["queries"] = [], []
        for k in range(case["sets"]):
            n = max(1, int(round(case["n"] * 2 ** -rng.uniform(0, 10))))
            nq = max(1, int(round(case["nq"] * 2 ** -rng.uniform(0, 10))))
            p, w, v = _sources(case, n, seed + 10 * k)
            st["trees"].append(sbh.sbh_build(p, w, v, leaf_size=case["leaf"]))
            st["queries"].append(_queries(case, p, nq, seed + 10 * k))
        st["out"] = torch.empty(sum(q.shape[0] for q in st["queries"]), device="cuda")
        st["plan"] = sbh.sbh_multi_plan_create(st["trees"], st["queries"], case["kernel"], case["S"], seed,
                                               outs=list(st["out"].split([q.shape[0] for q in st["queries"]])), **st["kw"])
        return st
    p, w, v = _sources(case, case["n"], seed)
    q = _queries(case, p, case["nq"], seed)
    if op == "host":
        st.update(p=p.cpu().pin_memory(), w=w.cpu().pin_memory(), v=None if v is None else v.cpu().pin_memory(),
                  q=q.cpu().pin_memory(), out=torch.empty(case["nq"]).pin_memory())
        return st
    st.update(p=p, w=w, v=v, q=q)
    if op in ("grad", "learned", "train", "bh"):
        st["tree"] = sbh.sbh_build(p, w, v, leaf_size=case["leaf"])
    if op == "grad":
        st["q"] = q.requires_grad_(True)
        st["go"] = torch.rand(case["nq"], device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed + 2)) + 0.5
    if op == "learned":
        st["net"] = sbh.sbh_mlp_create(seed)
        sbh.sbh_mlp_set_weights(st["net"], _proposal(seed))
    if op == "bh":
        sbh.sbh_eval_bh(st["tree"], q[:1], case["kernel"], case["theta"], **st["kw"])  # the 8-ary tree is kept too
    return st


def run(st):
    c, op, kw = st["case"], st["case"]["op"], st["kw"]
    if op == "step":
        tree = sbh.sbh_build(st["p"], st["w"], st["v"], leaf_size=c["leaf"])
        return sbh.sbh_eval(tree, st["q"], c["kernel"], c["S"], st["seed"], **kw)
    if op == "host":
        return sbh.sbh_solve_host(st["p"], st["w"], st["q"], st["v"], c["leaf"], c["kernel"], c["S"], st["seed"],
                                  out=st["out"], **kw)
    if op == "multi":
        sbh.sbh_multi_plan_launch(st["plan"])
        return st["out"]
    if op == "grad":
        out = sbh.StochasticSum(st["q"], st["tree"], c["kernel"], c["S"], st["seed"], **kw)
        return {"out": out, "grad": torch.autograd.grad(out, st["q"], st["go"])[0]}
    if op == "learned":
        return sbh.sbh_eval_learned(st["tree"], st["net"], st["q"], c["kernel"], c["S"], st["seed"], near=c["near"], **kw)
    if op == "train":
        net = sbh.sbh_mlp_create(st["seed"])
        loss = sbh.sbh_mlp_train(net, st["tree"], st["q"], c["kernel"], c["near"], c["steps"], **kw)
        return {"loss": loss, "weights": sbh.sbh_mlp_get_weights(net)[0]}
    if op == "bh":
        return sbh.sbh_eval_bh(st["tree"], st["q"], c["kernel"], c["theta"], c["vote"], **kw)
    if op == "bh_step":
        tree = sbh.sbh_build(st["p"], st["w"], st["v"], leaf_size=c["leaf"])
        return sbh.sbh_eval_bh(tree, st["q"], c["kernel"], c["theta"], c["vote"], **kw)
    if op == "brute":
        return sbh.sbh_eval_brute(st["p"], st["w"], st["q"], c["kernel"], st["v"], **kw)
    return sbh.sbh_eval_brute_grad(st["p"], st["w"], st["q"], c["kernel"], st["v"], **kw)


FLOPS = {"coulomb": 12, "winding": 18, "smoothdist": 16}  # of one term, a reciprocal root or exponential as one
TERMS = 350  # of one query and sample: control variates and the children of the swaps its paths take, about


def work(case):
    op, per = case["op"], FLOPS[case["kernel"]]
    vec = 7 if case["kernel"] == "winding" else 4
    n, nq = case.get("n", 0), case["nq"]
    if op == "multi":  # sizes are log-uniform over a factor of 2^10: their mean is 0.144 of the largest
        n, nq = 0.144 * case["sets"] * n, 0.144 * case["sets"] * nq
    size = 4.0 * vec * n + 16.0 * nq
    if op in ("grad", "brute_grad"):
        size, per = size + 12.0 * nq, 2 * per
    if op in ("brute", "brute_grad"):
        return {"bytes": size, "flops": per * n * nq}
    if op in ("bh", "bh_step"):  # well-separated nodes: a few hundred at theta = 0.8, ~ theta^-3
        return {"bytes": size, "flops": per * nq * 300.0 * (0.8 / case["theta"]) ** 3}
    if op == "train":  # rows of about 20 children at some hundred decisions of each query
        rows = 100.0 * 20 * nq
        return {"bytes": size + 28 * rows, "flops": case["steps"] * 6.0 * 1313 * rows + per * 50.0 * 0.02 * n * nq}
    return {"bytes": size, "flops": per * TERMS * nq * case["S"]}


# ---------------------------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------------------------
def exact(case, seed):
    """The exact sums (Eq. 1) and their gradients, in FP64. The estimates, Barnes-Hut and the trained
    weights have no value that could be given without the tree and the random stream they follow."""
    if case["op"] not in ("brute", "brute_grad") or case["n"] * case["nq"] > 1 << 36:
        return None
    st = prepare(case, seed)
    P, W, Q = st["p"].double(), st["w"].double(), st["q"].double()
    N = None if st["v"] is None else st["v"].double() * W[:, None]
    n, nq, kind = case["n"], case["nq"], case["kernel"]
    eps2 = float(np.float32(SOFTENING)) ** 2
    F = torch.zeros(nq, dtype=torch.float64, device="cuda")
    G = torch.zeros(nq, 3, dtype=torch.float64, device="cuda") if case["op"] == "brute_grad" else None
    block = max(1, (1 << 24) // n)
    for a in range(0, nq, block):
        q = Q[a:a + block]
        dx, dy, dz = (P[:, k][None, :] - q[:, k][:, None] for k in range(3))
        r2 = dx * dx
        r2.addcmul_(dy, dy).addcmul_(dz, dz)
        if kind == "coulomb":
            f = (r2.add_(eps2)).rsqrt_()
            F[a:a + block] = f @ W
            c = f.pow(3).mul_(W) if G is not None else None
        elif kind == "winding":
            dn = dx * N[:, 0]
            dn.addcmul_(dy, N[:, 1]).addcmul_(dz, N[:, 2])
            f = r2.rsqrt().masked_fill_(r2 == 0, 0.0)
            i3 = f.pow(3)
            F[a:a + block] = (dn * i3).sum(1) / (4 * math.pi)
            c = 3 * dn * i3 * f * f if G is not None else None
        else:
            d = r2.sqrt_()
            ref = d.amin(1)
            t = ((d - ref[:, None]) * -ALPHA).exp_().mul_(W)
            s = t.sum(1)
            F[a:a + block] = ref - s.log() / ALPHA
            c = -t / d.clamp_min(1e-300) / s[:, None] if G is not None else None  # d is -log(F) / alpha
        if G is not None:
            G[a:a + block] = torch.stack([(c * x).sum(1) for x in (dx, dy, dz)], 1)
            if kind == "winding":
                G[a:a + block] -= torch.stack([(i3 * N[:, k]).sum(1) for k in range(3)], 1)
                G[a:a + block] /= 4 * math.pi
    return F if G is None else (F, G)
