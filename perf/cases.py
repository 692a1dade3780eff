"""Timed cases of the framework: the calls a program makes, through the Python binding.

Evaluations of the dual and its gradient (dense and truncated, in the three precisions), a batch
of uneven problems, conditional centroids and transport maps, a whole solve, and the warm-start
network's inference and gradients.  Sizes are those of the repository's configurations and tests
(the unit square and cube meshes with their 3- and 4-point rules, Gaussian-mixture densities,
uniform or mixture targets) or lie between them.
"""
import math

import numpy as np
import torch

import paper_2507_23602_gb300 as rs

PRECISION = {"fp64": rs.FP64, "mixed": rs.MIXED, "compensated": rs.COMPENSATED}
IN_DIM, WIDTH = 18, 256           # the warm-start network: 16 density parameters and a 2-D target


def listed():
    return [
        # a handful of elements, as in a unit test or a coarse multilevel stage: launches and latency
        {"name": "eval small 2d mixed", "op": "eval", "d": 2, "mesh": 16, "n": 128, "eps": 2e-2,
         "precision": "mixed"},
        # the plain FP64 configuration: unit square, 64 x 64 x 2 triangles, 512 targets
        {"name": "eval square fp64", "op": "eval", "d": 2, "mesh": 64, "n": 512, "eps": 1e-2,
         "precision": "fp64"},
        # the FP64 reference evaluation of a cube of ordinary size
        {"name": "eval cube fp64", "op": "eval", "d": 3, "mesh": 16, "n": 16384, "eps": 1e-2,
         "precision": "fp64"},
        # an ordinary 2-D evaluation with ragged sizes, as inside an L-BFGS run
        {"name": "eval square ragged mixed", "op": "eval", "d": 2, "mesh": 101, "n": 5003,
         "eps": 5e-3, "precision": "mixed"},
        # the headline: dense evaluation of the 786,432 x 65,536 cube
        {"name": "eval cube mixed", "op": "eval", "d": 3, "mesh": 32, "n": 65536, "eps": 1e-3,
         "precision": "mixed"},
        # the same method truncated by the psi-aware cutoffs
        {"name": "tail cube mixed", "op": "tail", "d": 3, "mesh": 24, "n": 65536, "eps": 1e-3,
         "tail": 1e-12, "precision": "mixed"},
        # the reference evaluations that certify a mixed solve
        {"name": "eval cube compensated", "op": "eval", "d": 3, "mesh": 16, "n": 65536,
         "eps": 1e-3, "precision": "compensated"},
        # one round of the batched solver: uneven problems evaluated together
        {"name": "batch of 16", "op": "batch", "problems": 16, "nq_lo": 20000, "nq_hi": 200000,
         "n_lo": 1000, "n_hi": 16000},
        # the Lloyd step of the barycenter
        {"name": "centroids cube", "op": "centroids", "d": 3, "mesh": 16, "n": 4096, "eps": 2e-3},
        # a whole solve of a warm-start problem: eps-schedule, mixed iterations, certified stop
        {"name": "solve square", "op": "solve", "d": 2, "mesh": 64, "n": 4096, "eps": 5e-3},
        # the network's training step: 65,536 rows on the GPU
        {"name": "network gradients", "op": "gradients", "rows": 65536},
        # the network's prediction for one problem's 4,096 targets, host arrays as the caller has
        {"name": "network forward", "op": "forward", "rows": 4096},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["eval", "eval", "eval", "tail", "tail", "batch", "centroids", "maps",
                     "gradients", "forward"])
    if op in ("gradients", "forward"):
        return {"op": op, "rows": int(_log(rng, 512, 65536))}
    if op == "batch":
        return {"op": op, "problems": rng.randint(2, 16), "nq_lo": 20000,
                "nq_hi": int(_log(rng, 30000, 200000)), "n_lo": 1000,
                "n_hi": int(_log(rng, 2000, 16000))}
    precision = rng.choice(["fp64", "mixed", "compensated"]) if op in ("eval", "tail") else "mixed"
    d = rng.choice([2, 3])
    # points and targets: pairs up to the listed cases' of that precision
    mesh = int(round(_log(rng, 10, 180) if d == 2 else _log(rng, 5, 24)))
    nq = 6 * mesh ** 2 if d == 2 else 24 * mesh ** 3
    most = {"fp64": 1.6e9, "mixed": 2.1e10, "compensated": 6.4e9}[precision]
    n = int(_log(rng, 100, max(200.0, min(65536.0, most / nq))))
    case = {"op": op, "d": d, "mesh": mesh, "n": n, "eps": _log(rng, 1e-3, 5e-2)}
    if op in ("eval", "tail"):
        case["precision"] = precision
    if op == "tail":
        case["tail"] = rng.choice([1e-12, 1e-10, 1e-8])
    return case


# ---- inputs ------------------------------------------------------------------------------------

_MESHES = {}


def _mesh_points(d, mesh):
    """Quadrature points and weights of the unit square (two triangles a cell, 3 points each) or
    cube (six tetrahedra a cell, 4 points each), cell by cell, on the GPU."""
    if (d, mesh) not in _MESHES:
        if d == 2:
            corners = [[(0, 0), (1, 0), (1, 1)], [(0, 0), (1, 1), (0, 1)]]
            bary = np.full((3, 3), 1 / 6) + np.eye(3) / 2
        else:
            eye = np.eye(3, dtype=int)
            corners = [[np.zeros(3, int), eye[a], eye[a] + eye[b], np.ones(3, int)]
                       for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1))]
            s5 = math.sqrt(5.0)
            bary = np.full((4, 4), (5 - s5) / 20) + np.eye(4) * (4 * s5 / 20)
        inside = np.einsum("qa,cad->cqd", bary, np.array(corners, float)).reshape(-1, d)
        cells = np.stack(np.meshgrid(*[np.arange(mesh)] * d, indexing="ij"), -1).reshape(-1, d)
        x = ((cells[:, None, :] + inside[None]) / mesh).reshape(-1, d)
        if len(_MESHES) >= 4:
            _MESHES.clear()
        _MESHES[d, mesh] = torch.tensor(x, device="cuda")
    return _MESHES[d, mesh]


def _problem(d, mesh, n, rng, mixture_targets):
    """Points, normalised masses of a Gaussian-mixture density, targets and their weights."""
    x = _mesh_points(d, mesh)

    def mixture(k):
        return rng.uniform(0.15, 0.85, (k, d)), rng.uniform(0.1, 0.2, k)

    means, sigma = mixture(5 if d == 3 else 3)
    m = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for mu, s in zip(means, sigma):
        m += torch.exp(-0.5 * ((x - torch.tensor(mu, device="cuda")) ** 2).sum(1) / s ** 2) / s ** d
    m /= m.sum()
    if mixture_targets:
        means, sigma = mixture(4)
        at = rng.integers(0, 4, 4 * n)
        y = means[at] + sigma[at, None] * rng.standard_normal((4 * n, d))
        y = y[((y >= 0) & (y <= 1)).all(1)]
        y = np.concatenate([y, rng.uniform(0, 1, (max(0, n - len(y)), d))])[:n]
        nu = rng.uniform(0.5, 1.5, n)
    else:
        y, nu = rng.uniform(0, 1, (n, d)), np.ones(n)
    return x, m, torch.tensor(y, device="cuda"), torch.tensor(nu / nu.sum(), device="cuda")


def _single(case, seed):
    rng = np.random.default_rng(seed)
    x, m, y, nu = _problem(case["d"], case["mesh"], case["n"], rng, case["d"] == 3)
    psi = torch.tensor(0.005 * rng.standard_normal(case["n"]), device="cuda")
    return x, m, y, nu, psi


def _batch(case, seed):
    """Uneven 2-D and 3-D problems, eps log-uniform in [1e-3, 1e-1].  The sizes belong to the case;
    densities, targets and potentials to the seed."""
    sizes = np.random.default_rng(case["problems"] * 1000003 + case["nq_hi"] + case["n_hi"])
    rng = np.random.default_rng(seed)
    problems, eps = [], []
    for i in range(case["problems"]):
        d = 2 + i % 2
        nq = math.exp(sizes.uniform(math.log(case["nq_lo"]), math.log(case["nq_hi"])))
        n = int(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        mesh = round(math.sqrt(nq / 6)) if d == 2 else round((nq / 24) ** (1 / 3))
        eps.append(math.exp(sizes.uniform(math.log(1e-3), math.log(1e-1))))
        problems.append(_problem(d, mesh, n, rng, False))
    psi = 0.005 * rng.standard_normal(sum(p[2].shape[0] for p in problems))
    return problems, np.array(eps), psi


def _network(case, seed):
    """Parameters (weights of variance 1 / fan-in, small biases), rows and labels."""
    rng = np.random.default_rng(seed)
    pad = (IN_DIM + 31) // 32 * 32
    w1 = np.zeros((WIDTH, pad))
    w1[:, :IN_DIM] = rng.standard_normal((WIDTH, IN_DIM)) / math.sqrt(IN_DIM)
    square = [rng.standard_normal((WIDTH, WIDTH)) / math.sqrt(WIDTH) for _ in range(2)]
    bias = [0.1 * rng.standard_normal(WIDTH) for _ in range(3)]
    last = rng.standard_normal(WIDTH) / math.sqrt(WIDTH)
    params = np.concatenate([w1.ravel(), bias[0], square[0].ravel(), bias[1], square[1].ravel(),
                             bias[2], last, [0.0]]).astype(np.float32)
    x = rng.uniform(0, 1, (case["rows"], IN_DIM))
    x[:, 2:16:4] = np.log(0.1 + 0.1 * x[:, 2:16:4])
    x[:, 3:16:4] = 0.5 * rng.standard_normal((case["rows"], 4))
    return params, x.astype(np.float32), rng.standard_normal(case["rows"]).astype(np.float32)


# ---- the cases ---------------------------------------------------------------------------------

def prepare(case, seed):
    op = case["op"]
    if op in ("gradients", "forward"):
        params, x, y = _network(case, seed)
        net = rs.MLP(IN_DIM, WIDTH, seed=0)
        net.set_params(params)
        if op == "gradients":
            x, y = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
        return {"case": case, "net": net, "x": x, "y": y}
    if op == "batch":
        problems, eps, psi = _batch(case, seed)
        batch = rs.Batch([tuple(a.cpu().numpy() for a in p) for p in problems])
        return {"case": case, "batch": batch, "eps": eps, "psi": psi}
    x, m, y, nu, psi = _single(case, seed)
    state = {"case": case, "problem": rs.Problem(x, m, y, nu), "psi": psi}
    if op in ("eval", "tail"):
        state["grad"] = torch.empty_like(psi)
    return state


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "forward":
        return state["net"].forward(state["x"])
    if op == "gradients":
        return state["net"].gradients(state["x"], state["y"])
    if op == "batch":
        return state["batch"].eval(state["psi"], state["eps"])
    problem, psi = state["problem"], state["psi"]
    if op == "eval":
        return problem.eval(psi, case["eps"], 0.0, PRECISION[case["precision"]],
                            grad_out=state["grad"])
    if op == "tail":
        return problem.eval_tail(psi, case["eps"], case["tail"], PRECISION[case["precision"]],
                                 grad_out=state["grad"])
    if op == "centroids":
        return problem.centroids(psi, case["eps"])
    if op == "maps":
        return problem.transport_maps(psi, case["eps"])
    psi, stats = problem.solve(eps=case["eps"], eps_start=0.1, eps_factor=0.5, tol_l1=1e-6)
    return psi, stats.J


def work(case):
    op = case["op"]
    if op in ("gradients", "forward"):
        rows, layers = case["rows"], IN_DIM * WIDTH + 2 * WIDTH * WIDTH + WIDTH
        passes = 3 if op == "gradients" else 1
        return {"bytes": 4.0 * (rows * (IN_DIM + 1) + passes * layers),
                "flops": 2.0 * passes * rows * layers}
    if op == "batch":
        sizes = np.random.default_rng(case["problems"] * 1000003 + case["nq_hi"] + case["n_hi"])
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["problems"]):
            d = 2 + i % 2
            nq = math.exp(sizes.uniform(math.log(case["nq_lo"]), math.log(case["nq_hi"])))
            n = math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))
            sizes.uniform()
            total["bytes"] += 8.0 * (nq * (d + 1) + n * (d + 3))
            total["flops"] += nq * n * (4 * d + 6)
        return total
    d, n = case["d"], case["n"]
    nq = 6 * case["mesh"] ** 2 if d == 2 else 24 * case["mesh"] ** 3
    pairs = float(nq) * n
    data = 8.0 * (nq * (d + 1) + n * (d + 3))      # points, masses, targets, weights, psi, gradient
    if op == "tail":
        # the pairs within the cutoff radius of the bulk of the points
        r = math.sqrt(2 * case["eps"] * math.log(1 / case["tail"]))
        pairs *= min(1.0, math.pi * r ** 2 if d == 2 else 4 / 3 * math.pi * r ** 3)
    if op == "centroids":
        return {"bytes": data + 8.0 * n * d, "flops": pairs * (6 * d + 6)}
    if op == "maps":
        return {"bytes": data + 8.0 * nq * (d + 1), "flops": pairs * (4 * d + 4)}
    if op == "solve":
        return {"bytes": data, "flops": 60 * pairs * (4 * d + 6)}   # iterations of such a solve
    return {"bytes": data, "flops": pairs * (4 * d + 6)}


# ---- the same in 64 bits -----------------------------------------------------------------------

def _costs(x, y):
    c = torch.zeros((x.shape[0], y.shape[0]), dtype=torch.float64, device="cuda")
    for k in range(x.shape[1]):
        c.add_((x[:, k, None] - y[None, :, k]).square_(), alpha=0.5)
    return c


def _exact_sums(x, m, y, nu, psi, eps, tail=0.0, moments=False):
    """J, the gradient and the x-weighted sums of the plan, the points in chunks."""
    n, nq = y.shape[0], x.shape[0]
    a = psi / eps + torch.log(nu)
    mass = torch.zeros(n, dtype=torch.float64, device="cuda")
    first = torch.zeros((n, x.shape[1]), dtype=torch.float64, device="cuda")
    J = torch.zeros((), dtype=torch.float64, device="cuda")
    mean = torch.empty_like(x) if moments else None
    step = max(1, (1 << 26) // n)
    for q in range(0, nq, step):
        xq, mq = x[q:q + step], m[q:q + step]
        c = _costs(xq, y)
        s = torch.add(a[None, :], c, alpha=-1.0 / eps)
        if tail:
            near, at = c.min(1)
            alpha = near - psi[at] - eps * torch.log(nu[at])
            beta = psi + eps * math.log(1.0 / tail)
            s.masked_fill_(c >= alpha[:, None] + beta[None, :], -math.inf)
        del c
        top = s.max(1).values
        s.sub_(top[:, None]).exp_()
        total = s.sum(1)
        J += (mq * eps * (top + torch.log(total))).sum()
        s.mul_((mq / total)[:, None])
        mass += s.sum(0)
        if moments:
            first += s.T @ xq
            mean[q:q + step] = (s @ y) / mq[:, None]
    return J - (psi * nu).sum(), mass - nu, mass, first, mean


def exact(case, seed):
    op = case["op"]
    if op == "solve":       # the potential is determined by where the iteration stops
        return None
    if op in ("gradients", "forward"):
        params, x, y = _network(case, seed)
        p, x, y = (torch.tensor(v, device="cuda").double() for v in (params, x, y))
        pad = (IN_DIM + 31) // 32 * 32
        parts = list(torch.split(p, [WIDTH * pad, WIDTH, WIDTH * WIDTH, WIDTH, WIDTH * WIDTH, WIDTH,
                                     WIDTH, 1]))
        for k, cols in ((0, pad), (2, WIDTH), (4, WIDTH)):
            parts[k] = parts[k].reshape(WIDTH, cols)
        parts = [v.clone().requires_grad_(op == "gradients") for v in parts]
        h = torch.nn.functional.pad(x, (0, pad - IN_DIM))
        for k in (0, 2, 4):
            h = torch.nn.functional.silu(h @ parts[k].T + parts[k + 1])
        out = h @ parts[6] + parts[7]
        if op == "forward":
            return out
        loss = 0.5 * (out - y).square().mean()
        grads = torch.autograd.grad(loss, parts)
        return loss.detach(), torch.cat([g.reshape(-1) for g in grads])
    if op == "batch":
        problems, eps, psi = _batch(case, seed)
        psi = torch.tensor(psi, device="cuda")
        J, g, at = [], [], 0
        for (x, m, y, nu), e in zip(problems, eps):
            got = _exact_sums(x, m, y, nu, psi[at:at + y.shape[0]], e)
            J.append(got[0])
            g.append(got[1])
            at += y.shape[0]
        return torch.stack(J), torch.cat(g)
    x, m, y, nu, psi = _single(case, seed)
    if op == "tail":
        got = _exact_sums(x, m, y, nu, psi, case["eps"], case["tail"])
        return got[0], got[1], None
    J, g, mass, first, mean = _exact_sums(x, m, y, nu, psi, case["eps"],
                                          moments=op in ("centroids", "maps"))
    if op == "centroids":
        return first / nu[:, None], mass
    if op == "maps":
        return mean, None
    return J, g, x.shape[0] * y.shape[0]
