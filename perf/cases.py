"""Performance cases of the solver: scenario-tree SMPC solves as a control program runs them.

Every case is a solve through the C ABI's Python binding: a water network of the
flow-based model (tanks, actuators, junctions), a scenario tree or a forest of
trees on it, and a number of APG iterations that the sampling period allows.  The
sizes are those of the repository's workloads: the 15-node tiny tree, the single
scenario of certainty-equivalent MPC, the 2081- and 21111-node trees of the 63-tank
network, the uneven trees on networks of 20 to 63 tanks that are batched and served,
and ragged trees with random probabilities.

A case is a dict of plain values:
  groups     "n_x,n_u,n_d,n_e@tree;tree;..." joined by "/": one factor per group (a
             network with one tree, or a forest of trees); a tree is "N:AxBxC:S"
             (horizon, largest fan-outs of the first stages, scenarios) or "N:rMbK:T"
             (K random branching stages with 1..M children each, random probabilities, tree
             seed T)
  precision  fp64 | fp32 | bf16;  shared: one pack for all nodes (1) or one per node (0)
  entry      solve | static | batch | loop (a cold step, then a warm-started one)
  iters, graph, ergodic, dynamics (tank | leaky), scale (tiny | city)
"""
import math

import numpy as np
import torch

import paper_1604_01074_gb300 as smpc

PRECISION = {"fp64": smpc.SMPC_FP64, "fp32": smpc.SMPC_FP32, "bf16": smpc.SMPC_BF16}
BARCELONA = "63,114,88,17"


def _case(name, groups, precision, iters, **kw):
    return {**{"name": name, "groups": groups, "precision": precision, "shared": 0, "entry": "solve", "iters": iters,
               "graph": 1, "ergodic": 0, "dynamics": "tank", "scale": "city"}, **kw}


def listed():
    return [
        # the smallest call: a toy network's step, all launches and latency (500 iterations, Sec. V)
        _case("tiny_fp64", "4,6,3,1@4:2x2x2:8", "fp64", 500, graph=0, scale="tiny"),
        # certainty-equivalent MPC of the full network: one scenario, from a controller that may not allocate
        _case("ce_mpc_static_fp32", BARCELONA + "@24:1:1", "fp32", 60, entry="static", graph=0),
        # the paper's network with 100 scenarios in the precision that answers are checked against
        _case("barcelona_fp64", BARCELONA + "@24:5x5x2x2:100", "fp64", 60),
        # the same tree in the precision it is run in
        _case("barcelona_fp32", BARCELONA + "@24:5x5x2x2:100", "fp32", 60),
        # a middle-sized network on an irregular tree (late branchings, random probabilities), with the
        # ergodic average kept and one pack for all nodes
        _case("ragged_shared_fp32", "35,65,49,10@18:r4b4:26", "fp32", 100, shared=1, ergodic=1),
        # two closed-loop steps of the paper's second-largest class of controllers (242 scenarios):
        # a cold one, then one warm-started from its duals
        _case("closed_loop_fp32", BARCELONA + "@24:10x8x5:242", "fp32", 40, entry="loop"),
        # tanks that leak and exchange water: a general state matrix
        _case("leaky_fp32", "50,90,70,14@18:5x5x5:100", "fp32", 60, dynamics="leaky"),
        # the largest single tree (1000 scenarios): the headline solve, with a pack per node, with one
        # pack, and with 16-bit packs
        _case("large_fp32", BARCELONA + "@24:10x10x10:1000", "fp32", 60),
        _case("large_shared_fp32", BARCELONA + "@24:10x10x10:1000", "fp32", 60, shared=1),
        _case("large_bf16", BARCELONA + "@24:10x10x10:1000", "bf16", 60),
        # sixteen uneven trees on four networks in one batch, 16-bit shared packs
        _case("batch_shared_bf16",
              "20,40,28,6@24:7x7x7:301;12:3x3x3:22;18:6x6x6:199;12:8x8x8:460/"
              "35,65,49,10@18:8x8x8:411;24:5x5x5:97;12:6x6x6:163;24:4x4x4:50/"
              "50,90,70,14@12:8x8x8:487;18:7x7x7:260;24:3x3x3:19;12:6x6x6:150/"
              "63,114,88,17@24:8x8x8:380;12:5x5x5:101;18:5x5x5:120;18:7x7x7:333", "bf16", 60, shared=1, entry="batch"),
    ]


def draw(rng):
    """One more case: networks of 4 to 63 tanks, trees of 15 to 15000 nodes, every precision and option."""
    n_x = rng.choice([4, 7, 20, 35, 41, 50, 63])
    n_u = {4: 6, 7: 13}.get(n_x, int(1.8 * n_x) + rng.randrange(3))
    n_e = max(1, round(0.15 * n_u))
    n_d = max(n_e, round(1.4 * n_x) + rng.randrange(-2, 3))
    n_u = max(n_u, n_x + n_e)

    entry = rng.choice(["solve", "solve", "solve", "loop", "batch", "static"])
    leaky = entry == "solve" and rng.random() < 0.15
    precision = rng.choice(["fp32", "fp32", "fp64"] if leaky else ["fp64", "fp32", "fp32", "bf16"])

    def tree():
        N = rng.choice([7, 12, 18, 24])
        if rng.random() < 0.25:
            return "%d:r%db%d:%d" % (N, rng.randrange(2, 5), rng.randrange(1, 5), rng.randrange(1000))
        S = round(math.exp(rng.uniform(math.log(4), math.log(150 if precision == "fp64" else 500))))
        b = 2
        while b ** 3 < S:
            b += 1
        return "%d:%dx%dx%d:%d" % (N, b, b, b, max(S, b * b))

    groups = "%d,%d,%d,%d@" % (n_x, n_u, n_d, n_e)
    if entry == "batch":
        groups += ";".join(tree() for _ in range(rng.randrange(1, 5)))
    elif entry == "static":
        groups += "%d:%dx2:%d" % (rng.choice([8, 18, 24]), 4, rng.choice([5, 8]))
    else:
        groups += tree()
    iters = round(math.exp(rng.uniform(math.log(16), math.log(60)))) // (2 if entry == "loop" else 1)
    return {"groups": groups, "precision": precision, "shared": rng.randrange(2), "entry": entry,
            "iters": iters, "graph": 0 if entry == "static" else rng.randrange(2),
            "ergodic": int(entry in ("solve", "batch") and rng.random() < 0.2),
            "dynamics": "leaky" if leaky else "tank", "scale": "tiny" if n_x < 20 else "city"}


# ---------------------------------------------------------------- trees (from the case alone)
def _tree(text):
    """(parent, stage, probability) of one tree, nodes in breadth-first order."""
    N, shape, last = text.split(":")
    N, last = int(N), int(last)
    fans, width = [], 1
    if shape.startswith("r"):
        most, stages = (int(v) for v in shape[1:].split("b"))
        r = np.random.default_rng(last)
        branch = set(r.choice(N - 1, size=min(stages, N - 1), replace=False).tolist())
        for j in range(N - 1):
            fans.append(r.integers(1, most + 1, size=width) if j in branch else np.ones(width, dtype=np.int64))
            width = int(fans[-1].sum())
    else:
        b = [int(v) for v in shape.split("x")]
        for j in range(N - 1):
            if j < len(b) - 1:
                fan = np.full(width, b[j])
            elif j == len(b) - 1:  # near-even, reaching the scenario count exactly
                fan = np.full(width, last // width)
                fan[:last % width] += 1
            else:
                fan = np.ones(width, dtype=np.int64)
            fans.append(fan)
            width = int(fan.sum())
    parent, first, width = [np.array([-1])], 0, 1
    for fan in fans:
        parent.append(np.repeat(first + np.arange(width), fan))
        first, width = first + width, int(fan.sum())
    stage = np.concatenate([np.full(len(p), j) for j, p in enumerate(parent)])
    prob = [np.ones(1)]
    if shape.startswith("r"):
        for fan in fans:
            w = r.uniform(0.2, 1.0, size=int(fan.sum()))
            own = np.repeat(np.arange(len(fan)), fan)
            prob.append(prob[-1][own] * w / np.bincount(own, weights=w)[own])
    else:  # equiprobable scenarios
        leaves = [np.ones(width)]
        for fan in reversed(fans):
            leaves.append(np.bincount(np.repeat(np.arange(len(fan)), fan), weights=leaves[-1]))
        prob = [v / leaves[-1][0] for v in reversed(leaves)]
    return np.concatenate(parent).astype(np.int32), stage, np.concatenate(prob)


def _forest(texts):
    """Trees stacked stage by stage: parent, stage, prob, tree of every node, row of its stage's data, rows."""
    trees = [_tree(t) for t in texts]
    depth = [int(s[-1]) + 1 for _, s, _ in trees]
    off = np.concatenate([[0], np.cumsum(depth)])
    size = [len(p) for p, _, _ in trees]
    tree = np.repeat(np.arange(len(trees)), size)
    local = np.concatenate([np.arange(k) for k in size])
    stage = np.concatenate([s for _, s, _ in trees])
    order = np.lexsort((local, tree, stage))
    place = np.empty(len(order), dtype=np.int64)
    place[order] = np.arange(len(order))
    base = np.concatenate([[0], np.cumsum(size)])
    parent = np.concatenate([np.where(p < 0, -1, place[base[r] + np.maximum(p, 0)]) for r, (p, _, _) in enumerate(trees)])
    prob = np.concatenate([p for _, _, p in trees])
    tree, stage = tree[order], stage[order]
    return {"parent": parent[order].astype(np.int32), "stage": stage, "prob": prob[order], "tree": tree,
            "row": off[tree] + stage, "depth": depth, "trees": len(trees)}


# ---------------------------------------------------------------- networks and step data (from the seed)
def _network(rng, n_x, n_u, n_d, n_e, tiny, leaky):
    """A network whose junctions each have a supply that covers their worst demand."""
    dt = 1.0 if tiny else 3600.0
    src = np.full(n_u, -1)
    dst = np.concatenate([n_x + np.arange(n_e), np.arange(n_x), np.zeros(n_u - n_x - n_e, dtype=np.int64)])
    for a in range(n_e, n_u):
        if a < n_e + n_x:  # a supply into every tank, from a source or a junction
            src[a] = n_x + rng.integers(n_e) if n_e and rng.random() < 0.5 else -1
        else:  # links between tanks and junctions
            kind = rng.integers(3) if n_e else 0
            t, o = rng.choice(n_x, size=2, replace=False) if n_x > 1 else (0, 0)
            j = n_x + rng.integers(n_e) if n_e else -1
            src[a], dst[a] = ((t, o) if t != o else (-1, t), (t, j), (j, t))[kind]
    B, E = np.zeros((n_x, n_u)), np.zeros((n_e, n_u))
    for a in range(n_u):
        for node, sign in ((dst[a], 1.0), (src[a], -1.0)):
            if 0 <= node < n_x:
                B[node, a] += sign * dt
            elif node >= n_x:
                E[node - n_x, a] += sign
    at = np.concatenate([n_x + np.arange(n_e), np.where((rng.random(n_d - n_e) < 0.2) & (n_e > 0),
                                                       n_x + rng.integers(max(n_e, 1), size=n_d - n_e),
                                                       rng.integers(n_x, size=n_d - n_e))])
    Gd, Ed = np.zeros((n_x, n_d)), np.zeros((n_e, n_d))
    for i, node in enumerate(at):
        if node < n_x:
            Gd[node, i] = -dt
        else:
            Ed[node - n_x, i] = -1.0
    base = rng.uniform(0.5, 1.0, n_d) if tiny else rng.uniform(0.01, 0.1, n_d)
    cap = np.full(n_x, 10.0) if tiny else rng.uniform(500.0, 5000.0, n_x)
    u_max = rng.uniform(1.0, 3.0, n_u) if tiny else rng.uniform(0.5, 5.0, n_u)
    for j in range(n_e):
        u_max[j] = max(u_max[j], 2.0 * 1.69 * base[at == n_x + j].sum())
    A = np.eye(n_x)
    if leaky:  # tanks lose five percent a step and exchange three
        R = rng.uniform(0.0, 1.0, (n_x, n_x))
        np.fill_diagonal(R, 0.0)
        A = 0.95 * A + 0.03 * R / R.sum(axis=1, keepdims=True)
    net = {"A": A, "B": B, "Gd": Gd, "E": E, "Ed": Ed}
    cost = {"W_alpha": 1.0 if tiny else 2e4, "W_u": (1.0 if tiny else 1e5) * np.eye(n_u), "W_x": 10.0 if tiny else 1e7,
            "gamma_d": 100.0 if tiny else 5e7, "x_min": np.zeros(n_x), "x_max": cap, "x_s": 0.3 * cap,
            "u_min": np.zeros(n_u), "u_max": u_max,
            "alpha1": np.where(src < 0, rng.uniform(0.02, 0.1, n_u), 0.0)}
    return net, cost, base, at, np.where(rng.random(n_u) < 0.6, rng.uniform(0.01, 0.05, n_u), 0.0)


def _groups(case):
    for g in case["groups"].split("/"):
        sizes, trees = g.split("@")
        yield [int(v) for v in sizes.split(",")], trees.split(";")


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _problems(case, seed):
    """Network, tree, step data and plain 64-bit model of every group."""
    out = []
    for k, ((n_x, n_u, n_d, n_e), texts) in enumerate(_groups(case)):
        rng = np.random.default_rng([seed, k])
        tiny = case["scale"] == "tiny"
        net, cost, base, at, pump = _network(rng, n_x, n_u, n_d, n_e, tiny, case["dynamics"] == "leaky")
        T = _forest(texts)
        dhat, alpha2 = [], []
        for d in T["depth"]:
            t = int(rng.integers(24)) + np.arange(d)
            dhat.append((1.0 + 0.3 * np.sin(2 * np.pi * t / 24))[:, None] * base[None])
            alpha2.append(np.where((t % 24 >= 8) & (t % 24 < 20), 2.0, 1.0)[:, None] * (np.ones(n_u) if tiny else pump)[None])
        P = {"net": net, "cost": cost, "T": T, "dhat": np.concatenate(dhat), "alpha2": np.concatenate(alpha2)}
        P["p"] = [(rng.uniform(0.4, 0.8, (T["trees"], n_x)) * cost["x_max"]).reshape(-1) for _ in range(2)]
        q = np.zeros((T["trees"], n_u))
        for j in range(n_e):
            q[:, j] = [d[0][at == n_x + j].sum() for d in dhat]
        P["q"] = q.reshape(-1)
        dev = _device()
        gen = torch.Generator(device=dev).manual_seed(int(seed) * 64 + k)
        z = torch.randn((len(T["parent"]), n_d), dtype=torch.float64, device=dev, generator=gen).clamp_(-3, 3)
        P["eps"] = 0.1 * z * torch.from_numpy(P["dhat"]).to(dev)[torch.from_numpy(T["row"]).to(dev)]
        P["model"] = _Model(P)
        out.append(P)
    return out


# ---------------------------------------------------------------- the method in plain 64 bits
class _Model:
    """Factor step, Algorithm 1 and the APG iteration in float64 torch, a stage at a time."""

    def __init__(self, P):
        dev, T = _device(), P["T"]
        t = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).to(dev)  # noqa: E731
        self.P, self.t = P, t
        A, B, Gd, E, Ed = (P["net"][k] for k in ("A", "B", "Gd", "E", "Ed"))
        n_u = B.shape[1]
        L = np.linalg.svd(E)[2][E.shape[0]:].T if E.shape[0] else np.eye(n_u)
        Pu = -np.linalg.pinv(E) @ Ed if E.shape[0] else np.zeros((n_u, Gd.shape[1]))
        Rhat = P["cost"]["W_u"] @ L
        Rinv = np.linalg.inv(L.T @ Rhat)
        self.A, self.L, self.BL, self.Lam, self.Rhat = t(A), t(L), t(B @ L), t(-Rinv), t(Rhat)
        self.Pu, self.Pe = t(Pu), t(B @ Pu + Gd)
        self.prob = t(T["prob"])
        self.n, self.n_x, self.n_u = len(T["parent"]), B.shape[0], n_u
        ends = np.flatnonzero(np.diff(T["stage"])) + 1
        self.spans = list(zip([0, *ends], [*ends, self.n]))
        self.parent = torch.from_numpy(T["parent"].astype(np.int64)).to(dev)
        self.tree, self.row = torch.from_numpy(T["tree"]).to(dev), torch.from_numpy(T["row"]).to(dev)
        # Jacobi scaling of the dual (Sec. IV-D) in closed form along the paths
        S = 1.0 / (2.0 * self.prob)
        c0, c1, c2 = torch.zeros_like(S), torch.zeros_like(S), torch.zeros_like(S)  # sums of k^0, k^1, k^2 / (2 p)
        for j, (a, b) in enumerate(self.spans):
            if j:
                up = self.parent[a:b]
                c2[a:b] = c2[up] + 2 * c1[up] + c0[up]
                c1[a:b] = c1[up] + c0[up]
                c0[a:b] = c0[up]
            for c in (c0, c1, c2):
                c[a:b] += S[a:b]
        dB, dL = np.einsum("ij,jk,ik->i", B @ L, Rinv, B @ L), np.einsum("ij,jk,ik->i", L, Rinv, L)
        live = dL > 1e-12 * dL.max()
        dL = np.where(live, dL, dL[live].mean())
        self.d_x, self.d_u = 1.0 / (c2 * float(dB.mean())), 1.0 / (c0[:, None] * t(dL)[None])
        # largest eigenvalue of the scaled dual Hessian by power iteration
        gen = torch.Generator(device=dev).manual_seed(1)
        v = [torch.randn((self.n, k), dtype=torch.float64, device=dev, generator=gen) for k in (self.n_x, self.n_x, n_u)]
        sx, su = self.d_x.sqrt()[:, None], self.d_u.sqrt()
        top = 1.0
        for _ in range(16 if np.array_equal(A, np.eye(len(A))) else 80):
            norm = sum((a * a).sum() for a in v).sqrt()
            v = [a / norm for a in v]
            x, u = self.step(sx * (v[0] + v[1]), su * v[2])
            v = [-sx * x, -sx * x, -su * u]
            top = float(sum((a * a).sum() for a in v).sqrt())
        self.lam = float("%.6g" % (1.0 / (1.25 * top)))

    def step(self, xi, psi, data=None):
        """Algorithm 1: the primal iterate of the duals (linear part alone without data)."""
        s, r = xi.clone(), psi @ self.L
        if data:
            r += data["beta"]
        for j in range(len(self.spans) - 1, -1, -1):
            a, b = self.spans[j]
            r[a:b] += s[a:b] @ self.BL
            if j:
                up = self.spans[j - 1][0]
                s[up:a].index_add_(0, self.parent[a:b] - up, s[a:b] @ self.A)
                r[up:a].index_add_(0, self.parent[a:b] - up, r[a:b])
        v = (r @ self.Lam) / (2.0 * self.prob)[:, None]
        x = torch.zeros_like(xi)
        for j, (a, b) in enumerate(self.spans):
            if j:
                v[a:b] += v[self.parent[a:b]]
                x[a:b] = x[self.parent[a:b]] @ self.A.T
            elif data:
                x[a:b] = data["p"][self.tree[a:b]] @ self.A.T
            x[a:b] += v[a:b] @ self.BL.T
            if data:
                x[a:b] += data["e"][a:b]
        return x, v @ self.L.T + (data["uhat"] if data else 0.0)

    def data(self, p, q):
        P, t = self.P, self.t
        d = t(P["dhat"])[self.row] + P["eps"]
        uhat, pr = d @ self.Pu.T, self.prob[:, None]
        alpha = (t(P["cost"]["alpha1"])[None] + t(P["alpha2"])) @ self.L * P["cost"]["W_alpha"]
        roots = self.spans[0][1]
        up = torch.cat([t(q).reshape(-1, self.n_u), uhat[self.parent[roots:]]])
        D = pr * uhat - pr * up
        D.index_add_(0, self.parent[roots:], (pr * (uhat[self.parent.clamp(min=0)] - uhat))[roots:])
        return {"p": t(p).reshape(-1, self.n_x), "e": d @ self.Pe.T, "uhat": uhat,
                "beta": pr * alpha[self.row] + 2.0 * D @ self.Rhat}

    def solve(self, p, q, iters, y=None):
        """APG iterations (eq. apg-iteration): x, u, the duals and the ergodic averages."""
        c, t, data = self.P["cost"], self.t, self.data(p, q)
        lx, lu = self.lam * self.d_x[:, None], self.lam * self.d_u
        mu = self.prob[:, None] * c["W_x"]
        xs, lo, hi, ul, uh = (t(c[k]) for k in ("x_s", "x_min", "x_max", "u_min", "u_max"))
        if y is None:
            y = [torch.zeros((self.n, k), dtype=torch.float64, device=lx.device) for k in (self.n_x, self.n_x, self.n_u)]
        old, th0, th = y, 1.0, 1.0

        def dist(v, proj, most):  # prox of most * distance
            far = (v - proj).norm(dim=1, keepdim=True)
            return torch.where(far > most, v + most / far.clamp(min=1e-300) * (proj - v), proj)

        for k in range(iters):
            w = [a + th * (1.0 / th0 - 1.0) * (a - b) for a, b in zip(y, old)]
            x, u = self.step(w[0] + w[1], w[2], data)
            vs, vz, vp = w[0] / lx + x, w[1] / lx + x, w[2] / lu + u
            ts, tz = dist(vs, torch.maximum(vs, xs), mu / lx), dist(vz, vz.clamp(lo, hi), c["gamma_d"] / lx)
            old, y = y, [w[0] + lx * (x - ts), w[1] + lx * (x - tz), w[2] + lu * (u - vp.clamp(ul, uh))]
            bar = (x, u) if k == 0 else ((1 - th) * bar[0] + th * x, (1 - th) * bar[1] + th * u)
            th0, th = th, 0.5 * (math.sqrt(th ** 4 + 4 * th ** 2) - th ** 2)
        return x, u, y, bar


# ---------------------------------------------------------------- the measured path
class _Controller:
    """The handles and buffers a control program keeps."""

    def __init__(self, case, seed):
        self.case, self.problems, self.trees, self.facs, self.out, self.batch = case, [], [], [], [], None
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        for P in _problems(case, seed):
            M = P.pop("model")
            net = P["net"] if case["dynamics"] == "leaky" else {**P["net"], "A": None}
            self.trees.append(smpc.smpc_tree_create(P["T"]["parent"], P["T"]["prob"]))
            self.facs.append(smpc.smpc_factor(self.trees[-1], net, P["cost"], precision=PRECISION[case["precision"]],
                                              precondition=1, lam=M.lam, shared_packs=case["shared"]))
            new = lambda k: torch.zeros((M.n, k), dtype=dtype, device=P["eps"].device)  # noqa: B023, E731
            self.out.append({"u": new(M.n_u), "x": new(M.n_x), "y": new(2 * M.n_x + M.n_u)})
            if case["ergodic"]:
                self.out[-1].update(ubar=new(M.n_u), xbar=new(M.n_x))
            self.problems.append(P)
        self.u0 = np.zeros(self.problems[0]["T"]["trees"] * self.out[0]["u"].shape[1])
        if case["entry"] == "batch":
            self.batch = smpc.smpc_batch_create(self.facs)

    def __del__(self):
        if self.batch is not None:
            smpc.smpc_batch_destroy(self.batch)
        for f in self.facs:
            smpc.smpc_factor_destroy(f)
        for t in self.trees:
            smpc.smpc_tree_destroy(t)


def prepare(case, seed):
    return _Controller(case, seed)


def run(state):
    c = state.case
    common = {"max_iters": c["iters"], "check_every": 64, "stream": torch.cuda.current_stream()}
    if c["entry"] == "batch":
        steps = [{"p": P["p"][0], "q": P["q"], "dhat": P["dhat"], "alpha2": P["alpha2"], "eps": P["eps"].data_ptr()}
                 for P in state.problems]
        info = smpc.smpc_batch_solve(state.batch, steps, outputs=[(o["u"], o["x"], o["y"]) for o in state.out],
                                     bar_outputs=[(o["ubar"], o["xbar"]) for o in state.out] if c["ergodic"] else None,
                                     use_graph=c["graph"], ergodic=c["ergodic"], **common)
        return [state.out, [r["iterations"] for r in info]]
    P, o, fac = state.problems[0], state.out[0], state.facs[0]
    data = {"dhat": P["dhat"], "alpha2": P["alpha2"], "eps": P["eps"].data_ptr(), "u0_host": state.u0}
    if c["entry"] == "static":
        info = smpc.smpc_solve_static(fac, P["p"][0], P["q"], **data, **o, **common)
        return [o, info["iterations"]]
    info = smpc.smpc_solve(fac, P["p"][0], P["q"], use_graph=c["graph"], ergodic=c["ergodic"], **data, **o, **common)
    if c["entry"] == "loop":  # the next sampling period: measured state, the move just applied, warm duals
        info = smpc.smpc_solve(fac, P["p"][1], state.u0.copy(), use_graph=c["graph"], warm_start=1, **data, **o, **common)
    return [o, info["iterations"]]


def exact(case, seed):
    outs, its = [], []
    for P in _problems(case, seed):
        M, n = P["model"], case["iters"]
        x, u, y, bar = M.solve(P["p"][0], P["q"], n)
        if case["entry"] == "loop":
            x, u, y, bar = M.solve(P["p"][1], u[:P["T"]["trees"]].cpu().numpy().reshape(-1), n, y)
        outs.append({"u": u, "x": x, "y": torch.cat(y, dim=1)})
        if case["ergodic"]:
            outs[-1].update(ubar=bar[1], xbar=bar[0])
        its.append(n)
    return [outs, its] if case["entry"] == "batch" else [outs[0], its[0]]


def work(case):
    """One pass.  Per node and iteration: Lambda / (2 p_n) where every node has its own, the duals of two
    iterates in and one out (8 bytes an entry), the affine data, bounds' steps; 2 flops per entry of [Bbar; L]
    (twice) and Lambda.  What a chip's 129 MB of cache holds is read once in a pass, not once an iteration."""
    size = {"fp64": (8, 8), "fp32": (4, 4), "bf16": (2, 4)}[case["precision"]]
    nbytes = flops = outputs = 0.0
    for (n_x, n_u, n_d, n_e), texts in _groups(case):
        n = sum(len(_tree(t)[0]) for t in texts)
        n_v, n_k, nd = n_u - n_e, n_x + n_u, 2 * n_x + n_u
        flops += n * (2.0 * (2 * n_k * n_v + n_v * n_v) + 30 * nd)
        nbytes += n * ((0 if case["shared"] else n_v * n_v * size[0]) + 3 * 8 * nd + size[1] * (n_k + n_v + n_u))
        outputs += n * (size[1] * (n_k + nd) + 8 * n_d)
    passes = case["iters"] * (2 if case["entry"] == "loop" else 1)
    return {"bytes": nbytes * (passes if nbytes > 129e6 else 1) + outputs, "flops": flops * passes}
