"""Performance cases of the library: what a user's program has it do, over the
range of sizes it is used at.

A case is a dict of plain values; ``kind`` names the entry point:

  solve  ``Solver.set_rhs`` + ``Solver.solve`` of one domain from u = 0: the
         repeated solve of a fixed domain with new data (time stepping,
         parameter studies).  ``precision`` 0 is the plain FP64 cycle (the
         default), 1 the FP32 cycle inside FP64 refinement.
  host   ``Solver.solve_host``: the same solve with f, g and u in host memory.
  batch  ``Batch.solve`` of many star domains of uneven sizes, with new data
         set on every domain and every solution fetched.
  infer  ``cnn.Net.forward`` with the trained weights: the learned guess.
  train  ``cnn.Net.forward`` + ``cnn.Net.backward``: the gradient of a step.

Domains and network sizes are those of inputs.py, learn.py and the benchmark;
the seed draws the data (a manufactured solution with random amplitude, wave
numbers and phase; for the network, star domains with Gaussian sources).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1111_0983_gb300 import cnn, gcmg, inputs, learn

F64 = torch.float64


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest single solve in use: a Dirichlet disk on a 65^2 grid
        dict(name="disk65_fp64", kind="solve", domain="disk", n=65, nc=17, precision=0, rtol=1e-10),
        # an ordinary small mixed-boundary domain
        dict(name="star257_mixed", kind="solve", domain="star3", n=257, nc=33, precision=1, rtol=1e-10),
        # the benchmark's 2D workload in both forms
        dict(name="flower1025_mixed", kind="solve", domain="flower", n=1025, nc=33, precision=1, rtol=1e-10),
        dict(name="flower1025_fp64", kind="solve", domain="flower", n=1025, nc=33, precision=0, rtol=1e-10),
        # the largest 2D grid of the benchmark (1e-9: near the FP64 floor of that grid)
        dict(name="flower4097_mixed", kind="solve", domain="flower", n=4097, nc=33, precision=1, rtol=1e-9),
        # data in host memory, a coarsest grid that is no power of two
        dict(name="flower1409_host", kind="host", domain="flower", n=1409, nc=45, precision=1, rtol=1e-10),
        # 3D, from small to the largest that is quick to set up
        dict(name="torus129_fp64", kind="solve", domain="torus", n=129, nc=17, precision=0, rtol=1e-10),
        dict(name="torus257_mixed", kind="solve", domain="torus", n=257, nc=17, precision=1, rtol=1e-10),
        dict(name="torus385_mixed", kind="solve", domain="torus", n=385, nc=25, precision=1, rtol=1e-10),
        # many uneven domains at once (129^2 to 1025^2)
        dict(name="stars48_batch", kind="batch", first=0, count=48, rtol=1e-10),
        # the learned guess of one 513^2 problem, and a training batch of eight
        dict(name="guess513_infer", kind="infer", batch=1, n=513),
        dict(name="guess513x8_train", kind="train", batch=8, n=513),
    ]


def _grid(rng, lo, hi, ncs):
    """n = (nc - 1) 2^k + 1 near a size drawn evenly over the logarithm."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    nc = rng.choice(ncs)
    k = max(1, round(math.log2((want - 1) / (nc - 1))))
    while k > 1 and (nc - 1) * 2 ** k + 1 > hi:
        k -= 1
    return (nc - 1) * 2 ** k + 1, nc


def draw(rng):
    kind = rng.choice(["solve2", "solve2", "solve2", "solve3", "solve3", "host", "batch", "infer", "train"])
    if kind in ("solve2", "host"):
        domain, star = rng.choice(["disk", "flower", "flower", "star"]), rng.randint(0, 255)
        ncs = list(range(13, 26)) if domain == "disk" else list(range(33, 50))
        n, nc = _grid(rng, 65, 4097 if kind == "solve2" else 2049, ncs)
        if domain == "star":   # its own grid: a coarsest grid must resolve the drawn boundary
            domain, n, nc = "star%d" % star, inputs.star_params(star)["n"], 33
        return dict(kind="solve" if kind == "solve2" else "host", domain=domain, n=n, nc=nc,
                    precision=rng.choice([0, 1]) if kind == "solve2" else 1, rtol=1e-10 if n < 1500 else 1e-9)
    if kind == "solve3":
        precision = rng.choice([0, 1, 1])
        n, nc = _grid(rng, 65, 385 if precision else 193, list(range(17, 26)))
        return dict(kind="solve", domain="torus", n=n, nc=nc, precision=precision, rtol=1e-10)
    if kind == "batch":
        count = round(math.exp(rng.uniform(math.log(4), math.log(48))))
        return dict(kind="batch", first=rng.randint(0, 255 - count), count=count, rtol=1e-10)
    n = round(math.exp(rng.uniform(math.log(129), math.log(769))))
    return dict(kind=kind, batch=rng.randint(1, 4 if n > 513 else 8), n=n)


# ------------------------------------------------------------------- the data
def _problem(domain):
    if domain.startswith("star"):
        return inputs.star(int(domain[4:]))
    return {"disk": inputs.disk, "flower": inputs.flower, "torus": inputs.torus}[domain]()


class _Data:
    """u = A sin(a x + p) cos(b y + q) [e^{c z}] and its f = -Lap u, grad u."""

    def __init__(self, dim, seed):
        r = np.random.default_rng(seed)
        self.dim = dim
        self.A = r.uniform(0.5, 2.0)
        self.a, self.b = r.uniform(2.0, 4.0, 2)
        self.p, self.q = r.uniform(0.0, 2 * math.pi, 2)
        self.c = r.uniform(0.5, 1.0) if dim == 3 else 0.0

    def parts(self, X, m):
        """The factors sin, cos of both axes and the exponential, in module m's functions."""
        t, s = self.a * X[0] + self.p, self.b * X[1] + self.q
        e = m.exp(self.c * X[2]) if self.dim == 3 else 1.0
        return m.sin(t), m.cos(t), m.cos(s), m.sin(s), e

    def u(self, X, m=np):
        st, _, cs, _, e = self.parts(X, m)
        return self.A * st * cs * e

    def f(self, X, m=np):
        return (self.a ** 2 + self.b ** 2 - self.c ** 2) * self.u(X, m)

    def g(self, B, nu, types):
        """u at Dirichlet points, grad u . nu at Neumann points."""
        X = [B[:, k] for k in range(self.dim)]
        st, ct, cs, ss, e = self.parts(X, np)
        grad = [self.A * self.a * ct * cs * e, -self.A * self.b * st * ss * e]
        if self.dim == 3:
            grad.append(self.c * self.u(X))
        gn = sum(grad[k] * nu[:, k] for k in range(self.dim))
        return np.ascontiguousarray(np.where(types == 0, self.u(X), gn))

    def f_grid(self, n):
        x = -1.0 + torch.arange(n, dtype=F64, device="cuda") * (2.0 / (n - 1))
        X = [x.reshape([n if b == a else 1 for b in range(self.dim)]) for a in range(self.dim)]
        return self.f(X, torch).expand((n,) * self.dim).contiguous()


def _set_types(S, P):
    """Boundary types of every level; the finest level's ghosts and their types."""
    for l in range(S.nlev):
        G = S.ghosts(l)
        types = P.bc_types(G["B"])
        S.set_bc_types(l, types)
        if l == 0:
            fine = G, types
    return fine


def _star_input(i, n):
    """Network input [4][n][n] of learning domain i: level set, scaled source on
    the domain, boundary data (0) and the boundary-type mask at the ghosts."""
    P, f = learn.problem(i, n)
    phi = P.phi_grid(n)
    inside = phi < 0
    near = np.zeros_like(inside)
    for axis in (0, 1):
        for step in (1, -1):
            near |= np.roll(inside, step, axis)
    ghost = near & ~inside
    X = inputs.coords(2, n)
    neumann = P.is_neumann(np.stack([X[0].ravel(), X[1].ravel()], 1)).reshape(n, n)
    x = np.zeros((4, n, n), np.float32)
    x[0] = phi
    x[1] = np.where(inside, f / learn.F_SCALE, 0.0)
    x[3] = np.where(ghost, np.where(neumann, -1.0, 1.0), 0.0)
    return x


def _net_inputs(case, seed):
    """(parameters, input batch, dL/dout) of a network case, on the host."""
    r = np.random.default_rng(seed)
    b, n = case["batch"], case["n"]
    first = 10 ** 6 + int(r.integers(0, 10 ** 6))
    x = np.stack([_star_input(first + k, n) for k in range(b)])
    if case["kind"] == "infer":
        params = learn.load_weights()
        return params, x, None
    parts = [(r.standard_normal((co, ci, 3, 3)) * math.sqrt(2.0 / (9 * ci)), 0.1 * r.standard_normal(co))
             for ci, co in cnn.LAYERS]
    # the derivative of a mean squared error against a smooth solution on the domain (channel 1 is not trained)
    X = inputs.coords(2, n)
    dout = np.zeros((b, 2, n, n), np.float32)
    for k in range(b):
        dout[k, 0] = np.where(x[k, 0] < 0, -2.0 * _Data(2, int(r.integers(1 << 30))).u(X), 0.0) / (b * n * n)
    return cnn.pack_params(parts), x, dout


# ------------------------------------------------------------------- one pass
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "host"):
        P, n = _problem(case["domain"]), case["n"]
        data = _Data(P.dim, seed)
        S = gcmg.Solver(P.phi_grid(n), case["nc"], precision=case["precision"], rtol=case["rtol"])
        G, types = _set_types(S, P)
        f, g = data.f_grid(n), torch.from_numpy(data.g(G["B"], G["nu"], types))
        if kind == "host":
            u = torch.empty((n,) * P.dim, dtype=F64, pin_memory=True)
            return dict(kind=kind, S=S, f=f.cpu().pin_memory().numpy(), g=g.pin_memory().numpy(), u=u.numpy())
        return dict(kind=kind, S=S, f=f, g=g.cuda(), u=torch.empty((n,) * P.dim, dtype=F64, device="cuda"))
    if kind == "batch":
        probs = [inputs.star(case["first"] + k) for k in range(case["count"])]
        sizes = [P.meta["n"] for P in probs]
        B = gcmg.Batch([P.phi_grid(n) for P, n in zip(probs, sizes)], 33, rtol=case["rtol"])
        fs, gs, us = [], [], []
        for k, (S, P, n) in enumerate(zip(B.domains, probs, sizes)):
            data = _Data(2, seed * 1000 + k)
            G, types = _set_types(S, P)
            fs.append(data.f_grid(n))
            gs.append(torch.from_numpy(data.g(G["B"], G["nu"], types)).cuda())
            us.append(torch.empty((n, n), dtype=F64, device="cuda"))
        return dict(kind=kind, B=B, f=fs, g=gs, u=us)
    params, x, dout = _net_inputs(case, seed)
    net = cnn.Net(case["batch"], case["n"], case["n"])
    net.set_params(params)
    state = dict(kind=kind, net=net, x=torch.from_numpy(x).cuda(),
                 out=torch.empty((case["batch"], 2, case["n"], case["n"]), device="cuda"))
    if kind == "train":
        state["dout"] = torch.from_numpy(dout).cuda()
        state["grad"] = torch.empty(cnn.num_params(), device="cuda")
    return state


def run(state):
    kind = state["kind"]
    if kind == "solve":
        state["S"].set_rhs(state["f"], state["g"])
        stats = state["S"].solve(state["u"].zero_())
        return dict(u=state["u"], converged=stats["converged"])
    if kind == "host":
        u, stats = state["S"].solve_host(state["f"], state["g"], state["u"])
        return dict(u=u, converged=stats["converged"])
    if kind == "batch":
        B = state["B"]
        for S, f, g in zip(B.domains, state["f"], state["g"]):
            S.set_rhs(f, g)
        stats, _ = B.solve()
        for k, u in enumerate(state["u"]):
            B.solution(k, u)
        return dict(u=state["u"], converged=all(s["converged"] for s in stats))
    state["net"].forward(state["x"], state["out"])
    if kind == "infer":
        return state["out"]
    state["net"].backward(state["dout"], state["grad"])
    return dict(out=state["out"], grad=state["grad"])


# ------------------------------------------------------------- what it takes
def _unknowns(P, n):
    """|Omega_h| from the level set's share of a coarser sampling of the box."""
    m = 257 if P.dim == 2 else 65
    return float((P.phi_grid(min(n, m)) < 0).mean()) * n ** P.dim


def work(case):
    """Inputs read once and outputs written once.  Operations of a solve: ten
    V(2,1) cycles (a factor of 0.1 each), per cycle and unknown three sweeps, a
    defect and the transfers, over all levels; of the network: its products."""
    kind = case["kind"]
    if kind in ("infer", "train"):
        px = case["batch"] * case["n"] ** 2
        mac = 9 * sum(ci * co for ci, co in cnn.LAYERS)
        later = 9 * sum(ci * co for ci, co in cnn.LAYERS[1:])   # gradients to the inputs of layers 2-6
        flops = 2 * px * (mac if kind == "infer" else 2 * mac + later)
        return dict(bytes=px * 4 * (6 if kind == "infer" else 8), flops=flops)
    if kind == "batch":
        doms = [(inputs.star(case["first"] + k), inputs.star_params(case["first"] + k)["n"])
                for k in range(case["count"])]
    else:
        doms = [(_problem(case["domain"]), case["n"])]
    total = dict(bytes=0.0, flops=0.0)
    for P, n in doms:
        m = _unknowns(P, n)
        per_cycle = (3 * (2 * P.dim + 2) + (2 * P.dim + 3) + 16) * (4.0 / 3 if P.dim == 2 else 8.0 / 7)
        total["bytes"] += 8 * m + 8 * n ** P.dim
        total["flops"] += 10 * per_cycle * m
    return total


# ------------------------------------------------------------------ in 64 bits
def _dense_disk(n, data):
    """Direct solution of the discrete Dirichlet problem on the disk: 5-point
    rows at the inside nodes; at each ghost the interpolation at the closest
    boundary point on the upwind 3 x 3 nodes, or, where one of them is no
    unknown, the first of 2 x 2, corner and two-point that has all its nodes.
    None if a ghost's offset vanishes along an axis."""
    P, h = inputs.disk(), 2.0 / (n - 1)
    phi = P.phi_grid(n)
    inside = phi < 0
    near = np.zeros_like(inside)
    for axis in (0, 1):
        for step in (1, -1):
            near |= np.roll(inside, step, axis)
    known = near | inside
    number = -np.ones((n, n), np.int64)
    number[known] = np.arange(known.sum())
    A = np.zeros((int(known.sum()),) * 2)
    b = np.zeros(A.shape[0])
    I, J = np.nonzero(inside)
    rows = number[I, J]
    A[rows, rows] = 4 / h ** 2
    for di, dj in ((1, 0), (-1, 0), (0, 1), (0, -1)):
        A[rows, number[I + di, J + dj]] = -1 / h ** 2
    b[rows] = data.f([-1 + I * h, -1 + J * h])
    for i, j in zip(*np.nonzero(near & ~inside)):
        grad = [(phi[i + 1, j] - phi[i - 1, j]) / (2 * h), (phi[i, j + 1] - phi[i, j - 1]) / (2 * h)]
        d = [-phi[i, j] * c / (grad[0] ** 2 + grad[1] ** 2) for c in grad]
        if d[0] == 0 or d[1] == 0:
            return None
        s = [1 if c > 0 else -1 for c in d]
        t = [d[k] / (s[k] * h) for k in range(2)]
        quad = [[(v - 1) * (v - 2) / 2, v * (2 - v), v * (v - 1) / 2] for v in t]
        rules = [{(k * s[0], m * s[1]): quad[0][k] * quad[1][m] for k in range(3) for m in range(3)},
                 {(k * s[0], m * s[1]): [1 - t[0], t[0]][k] * [1 - t[1], t[1]][m] for k in range(2) for m in range(2)},
                 {(0, 0): 1 - t[0] - t[1], (s[0], 0): t[0], (0, s[1]): t[1]}]
        for axis in (0, 1):   # towards the first inside neighbour
            for sg in (-1, 1):
                o = (sg, 0) if axis == 0 else (0, sg)
                if inside[i + o[0], j + o[1]]:
                    rules.append({(0, 0): 1 - d[axis] / (sg * h), o: d[axis] / (sg * h)})
        rule = next(w for w in rules if all(known[i + a, j + c] for a, c in w))
        for (a, c), w in rule.items():
            A[number[i, j], number[i + a, j + c]] += w
        b[number[i, j]] = data.u([-1 + i * h + d[0], -1 + j * h + d[1]])
    u = np.zeros((n, n))
    u[known] = np.linalg.solve(A, b)
    return u


def exact(case, seed):
    """Direct solutions of the small Dirichlet problems (larger ones take a
    sparse solver) and the network in FP64."""
    kind = case["kind"]
    if kind in ("solve", "host"):
        if case["domain"] != "disk" or case["n"] > 129:
            return None
        u = _dense_disk(case["n"], _Data(2, seed))
        return None if u is None else dict(u=u, converged=None)
    if kind == "batch":
        return None
    params, x, dout = _net_inputs(case, seed)
    y = torch.from_numpy(x).cuda().double()
    weights = []
    for l, (w, b) in enumerate(cnn.unpack_params(params)):
        w, b = (torch.from_numpy(v).cuda().double().requires_grad_(kind == "train") for v in (w, b))
        weights += [w, b]
        d = cnn.DILATIONS[l]
        y = torch.nn.functional.conv2d(y, w, b, padding=d, dilation=d)
        if l + 1 < len(cnn.LAYERS):
            y = torch.relu(y)
    if kind == "infer":
        return y
    grads = torch.autograd.grad(y, weights, torch.from_numpy(dout).cuda().double())
    return dict(out=y.detach(), grad=torch.cat([v.reshape(-1) for v in grads]))
